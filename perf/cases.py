"""Timed workloads of the triangle counter, through its public Python entry points.

Every case is one call (or one short sequence of calls) that a program makes on
a graph it holds: counting a device-resident CSR, building the CSR from edge
tuples, uploading and counting a host CSR, per-vertex counts, listing, and one
batch of many small graphs.  Graph families and sizes follow the benchmark and
the tests: R-MAT (edge factor 16, A/B/C/D = .57/.19/.19/.05), Chung-Lu power
laws (gamma 2.1, mean degree 32), uniform random graphs, grids with random
diagonals (road-like), and the mixed batch (n log-uniform in [64, 65536]).

Inputs are drawn on the GPU from the seed alone, with plain torch operations.
"""
from __future__ import annotations

import math

import torch

import paper_2309_09064_gb300 as tc

DEV = "cuda:0"


def listed():
    return [
        # an ego network or a subgraph of a query: latency and launches count
        dict(name="count_rmat10", kind="count", family="rmat", scale=10, degree=16.0, order="degree", levels=False),
        # a mid-sized social graph whose BFS levels the caller wants too
        dict(name="levels_rmat16", kind="count", family="rmat", scale=16, degree=16.0, order="degree", levels=True),
        # a social graph of a million vertices
        dict(name="count_rmat20", kind="count", family="rmat", scale=20, degree=16.0, order="degree", levels=False),
        # the benchmark's graph: 16.8 M vertices, 260 M edges
        dict(name="count_rmat24", kind="count", family="rmat", scale=24, degree=16.0, order="degree", levels=False),
        # a power-law web or citation graph, vertex count not a power of two
        dict(name="count_power4m", kind="count", family="power", n=4194301, degree=32.0, order="degree", levels=False),
        # near-uniform degrees: contact or similarity graphs, few triangles
        dict(name="count_uniform1m", kind="count", family="uniform", n=1048573, degree=32.0, order="degree",
             levels=False),
        # a road network: low degrees, thousands of BFS levels
        dict(name="count_grid", kind="count", family="grid", rows=4096, cols=4096, order="degree", levels=False),
        # the input step: raw edge tuples (loops, repeats, both directions) to a CSR
        dict(name="build_rmat21", kind="build", family="rmat", scale=21, degree=16.0),
        # the whole request: a CSR in pinned host memory, copied, counted, released
        dict(name="upload_rmat21", kind="upload", family="rmat", scale=21, degree=16.0, order="degree"),
        # clustering coefficients: triangles through every vertex
        dict(name="vertices_rmat19", kind="vertices", family="rmat", scale=19, degree=16.0, order="degree"),
        # every triangle written out, then put in canonical order
        dict(name="list_rmat16", kind="list", family="rmat", scale=16, degree=16.0, order="degree"),
        # many small independent graphs in one call
        dict(name="batch_512", kind="batch", graphs=512, n_lo=64, n_hi=65536),
    ]


def draw(rng):
    """One more case of the same ranges."""
    def log_int(lo, hi):
        return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    kind = rng.choice(["count", "count", "count", "count", "count", "build", "upload", "vertices", "list", "batch"])
    if kind == "batch":
        return dict(kind="batch", graphs=log_int(16, 512), n_lo=64, n_hi=log_int(4096, 65536))
    top = {"count": 22, "build": 21, "upload": 21, "vertices": 19, "list": 16}[kind]
    case = dict(kind=kind)
    family = rng.choice(["rmat", "rmat", "power", "uniform", "grid"])
    case["family"] = family
    if family == "rmat":
        case.update(scale=rng.randint(9, top), degree=round(rng.uniform(6.0, 20.0), 3))
    elif family == "grid":
        side = int(2 ** (top / 2))
        case.update(rows=log_int(30, side), cols=log_int(30, side) | 1)
    else:
        case.update(n=log_int(500, 1 << (top if kind != "list" else 15)) | 1, degree=round(rng.uniform(4.0, 40.0), 3))
    if kind != "build":
        # the id order is the working order of graphs whose numbering is kept for locality
        case["order"] = "id" if family in ("grid", "uniform") and rng.random() < 0.3 else "degree"
    if kind == "count":
        case["levels"] = rng.random() < 0.3
    return case


# ----------------------------------------------------------------------------- graphs

def _rmat(scale, tuples, gen):
    """R-MAT tuples with permuted vertex ids."""
    src = torch.zeros(tuples, dtype=torch.int32, device=DEV)
    dst = torch.zeros(tuples, dtype=torch.int32, device=DEV)
    u = torch.empty(tuples, dtype=torch.float32, device=DEV)
    for _ in range(scale):
        u.uniform_(generator=gen)
        low = u >= 0.76           # lower half: C or D
        right = ((u >= 0.57) & ~low) | (u >= 0.95)
        src.mul_(2).add_(low)
        dst.mul_(2).add_(right)
    perm = torch.randperm(1 << scale, generator=gen, device=DEV, dtype=torch.int64).to(torch.int32)
    return perm[src.long()], perm[dst.long()]


def _power(n, mean, gen):
    """Chung-Lu tuples, gamma = 2.1, weights capped at the square root of their sum."""
    w = (torch.arange(n, device=DEV, dtype=torch.float64) + 1.0).pow_(-1.0 / 1.1)
    w *= mean * n / w.sum()
    w.clamp_(max=math.sqrt(mean * n))
    cdf = torch.cumsum(w, 0)
    t = int(mean * n / 2)
    ends = []
    perm = torch.randperm(n, generator=gen, device=DEV, dtype=torch.int64).to(torch.int32)
    for _ in range(2):
        x = torch.rand(t, generator=gen, device=DEV, dtype=torch.float64) * cdf[-1]
        ends.append(perm[torch.searchsorted(cdf, x).clamp_(max=n - 1)])
    return ends[0], ends[1]


def _grid(rows, cols, gen):
    """Grid edges plus one random diagonal per cell with probability 0.3, row-major ids."""
    ids = torch.arange(rows * cols, device=DEV, dtype=torch.int32).view(rows, cols)
    diag = torch.rand((rows - 1, cols - 1), generator=gen, device=DEV) < 0.3
    back = torch.rand((rows - 1, cols - 1), generator=gen, device=DEV) < 0.5
    down, anti = diag & ~back, diag & back
    a = [ids[:, :-1].reshape(-1), ids[:-1].reshape(-1), ids[:-1, :-1][down], ids[:-1, 1:][anti]]
    b = [ids[:, 1:].reshape(-1), ids[1:].reshape(-1), ids[1:, 1:][down], ids[1:, :-1][anti]]
    return torch.cat(a), torch.cat(b)


def _tuples(case, gen):
    """(n, src, dst): raw edge tuples, int32 on the GPU."""
    f = case["family"]
    if f == "rmat":
        return (1 << case["scale"],) + _rmat(case["scale"], int(case["degree"] * (1 << case["scale"])), gen)
    if f == "power":
        return (case["n"],) + _power(case["n"], case["degree"], gen)
    if f == "uniform":
        t = int(case["degree"] * case["n"] / 2)
        pick = lambda: torch.randint(0, case["n"], (t,), generator=gen, device=DEV, dtype=torch.int32)
        return case["n"], pick(), pick()
    return (case["rows"] * case["cols"],) + _grid(case["rows"], case["cols"], gen)


def _csr(n, src, dst):
    """Simple undirected CSR of the tuples: (row_ptr int64[n + 1], col int32)."""
    keep = src != dst
    a, b = src[keep].long(), dst[keep].long()
    key = torch.cat([a * n + b, b * n + a])
    del a, b, keep
    key = torch.sort(key).values
    first = torch.ones_like(key, dtype=torch.bool)
    first[1:] = key[1:] != key[:-1]
    key = key[first]
    rp = torch.searchsorted(key, torch.arange(n + 1, device=DEV, dtype=torch.int64) * n)
    return rp, key.remainder_(n).to(torch.int32)


def _batch_graphs(case, gen):
    """CSRs of the mixed batch: n log-uniform, R-MAT (edge factor 8..32) or uniform (mean degree 4..64)."""
    u = torch.rand((case["graphs"], 3), generator=gen, device=DEV, dtype=torch.float64).tolist()
    lo, hi = case["n_lo"], case["n_hi"]
    for x, coin, y in u:
        n = max(lo, min(hi, int(lo * (hi / lo) ** x)))
        if coin < 0.5:
            scale = n.bit_length() - 1
            n = 1 << scale
            src, dst = _rmat(scale, (8 + int(25 * y)) * n, gen)
        else:
            t = int((4.0 + 60.0 * y) * n / 2)
            src, dst = (torch.randint(0, n, (t,), generator=gen, device=DEV, dtype=torch.int32) for _ in range(2))
        yield (n,) + _csr(n, src, dst)


def _generator(seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed))
    return gen


# ----------------------------------------------------------------------------- the calls

class _Library:
    """A context and the graphs made on it; released together."""

    def __init__(self, order="degree"):
        self.ctx = tc.tc_create(0, order=tc.TC_ORDER_ID if order == "id" else tc.TC_ORDER_DEGREE)
        self.graphs = []

    def borrow(self, rp, col):
        self.graphs.append(tc.tc_graph_from_csr(self.ctx, rp, col, tc.TC_BORROW))
        return self.graphs[-1]

    def __del__(self):
        for g in self.graphs:
            tc.tc_graph_free(g)
        tc.tc_destroy(self.ctx)


class _View:
    """Device memory of the library as an array that torch can wrap (while the graph lives)."""

    def __init__(self, address, count, kind):
        self.__cuda_array_interface__ = dict(shape=(count,), typestr=kind, data=(address, False), version=2)


def _copy_from(buffer, address, count, kind):
    """The library's array of `count` numbers into the first places of a torch buffer."""
    if count:
        buffer[:count].copy_(torch.as_tensor(_View(address, count, kind), device=DEV))


def _capacity(case):
    """Room for the triangles of a case of this size, whatever the seed."""
    return int(0.15 * _size(case)[1] ** (4.0 / 3.0)) + 100_000


def prepare(case, seed):
    gen = _generator(seed)
    kind = case["kind"]
    lib = _Library(case.get("order", "degree"))
    state = dict(kind=kind, lib=lib)
    if kind == "batch":
        state["csr"] = list(_batch_graphs(case, gen))
        torch.cuda.synchronize()
        state["graphs"] = [lib.borrow(rp, col) for _, rp, col in state["csr"]]
        return state
    n, src, dst = _tuples(case, gen)
    if kind == "build":
        state.update(n=n, src=src, dst=dst, row_ptr=torch.zeros(n + 1, dtype=torch.int64, device=DEV),
                     col=torch.zeros(2 * src.numel(), dtype=torch.int32, device=DEV))
        torch.cuda.synchronize()
        return state
    rp, col = _csr(n, src, dst)
    del src, dst
    if kind == "upload":
        state["rp"], state["col"] = rp.cpu().pin_memory(), col.cpu().pin_memory()
        return state
    state["csr"] = (rp, col)
    torch.cuda.synchronize()
    g = state["graph"] = lib.borrow(rp, col)
    if kind == "vertices":
        state["counts"] = torch.empty(n, dtype=torch.int64, device=DEV)
    elif kind == "list":
        state["triples"] = torch.empty(3 * _capacity(case), dtype=torch.int32, device=DEV)
        state["keys"] = torch.zeros(_capacity(case), dtype=torch.int64, device=DEV)
    elif case["levels"]:
        state["levels"] = torch.empty(n, dtype=torch.int32, device=DEV)
    return state


def _counts(T, stats):
    return dict(triangles=T, t_same=stats["t_same"], t_cross=stats["t_cross"],
                horizontal_edges=stats["horizontal_edges"], levels=stats["levels"], components=stats["components"])


def _canonical(triples):
    """The listed triangles as sorted keys a << 42 | b << 21 | c, a < b < c (ids below 2^21)."""
    x, y, z = triples.view(-1, 3).unbind(1)
    lo, hi = torch.minimum(x, y), torch.maximum(x, y)
    a, c = torch.minimum(lo, z), torch.maximum(hi, z)
    b = torch.maximum(lo, torch.minimum(hi, z))
    return torch.sort((a.long() << 42) | (b.long() << 21) | c).values


def run(state):
    kind, ctx = state["kind"], state["lib"].ctx
    if kind == "count":
        if "levels" in state:
            T, stats = tc.tc_count_levels(ctx, state["graph"], state["levels"])
            return dict(_counts(T, stats), L=state["levels"])
        return _counts(*tc.tc_count(ctx, state["graph"]))
    if kind == "build":
        # the program keeps the CSR in arrays of its own and gives the library's back
        g = tc.tc_build_csr(ctx, state["n"], state["src"], state["dst"])
        n, slots, rp, col = tc.tc_graph_info(g)
        _copy_from(state["row_ptr"], rp, n + 1, "<i8")
        _copy_from(state["col"], col, slots, "<i4")
        torch.cuda.current_stream().synchronize()  # the graph's memory is read until here
        tc.tc_graph_free(g)
        return dict(row_ptr=state["row_ptr"], col=state["col"], slots=slots)
    if kind == "upload":
        g = tc.tc_graph_from_csr(ctx, state["rp"], state["col"])
        T, stats = tc.tc_count(ctx, g)
        tc.tc_graph_free(g)
        return _counts(T, stats)
    if kind == "vertices":
        T, stats = tc.tc_count_vertices(ctx, state["graph"], state["counts"])
        return dict(_counts(T, stats), counts=state["counts"])
    if kind == "list":
        T, stats = tc.tc_list_triangles(ctx, state["graph"], state["triples"], state["triples"].numel() // 3)
        state["keys"][:T] = _canonical(state["triples"][:3 * T])
        return dict(_counts(T, stats), triples=state["keys"])
    return dict(counts=tc.tc_count_batch(ctx, state["graphs"]).astype("int64"))


# ----------------------------------------------------------------------------- what a pass needs at least

def _size(case):
    """(vertices, CSR slots) of a case, the slots from the tuples drawn (repeats left in)."""
    f = case["family"]
    if f == "rmat":
        n = 1 << case["scale"]
        return n, 2 * int(case["degree"] * n)
    if f == "grid":
        r, c = case["rows"], case["cols"]
        return r * c, 2 * int(r * (c - 1) + (r - 1) * c + 0.3 * (r - 1) * (c - 1))
    return case["n"], 2 * int(case["degree"] * case["n"] / 2)


def work(case):
    """The CSR read once (tuples for a build), the results written once; no arithmetic but compares."""
    kind = case["kind"]
    if kind == "batch":
        # mean n of a log-uniform size, about 36 slots per vertex
        lo, hi = case["n_lo"], case["n_hi"]
        n = (hi - lo) / math.log(hi / lo) * case["graphs"]
        return dict(bytes=8 * n + 4 * 36 * n + 8 * case["graphs"], flops=0)
    n, slots = _size(case)
    csr = 8 * (n + 1) + 4 * slots
    if kind == "build":
        return dict(bytes=4 * slots + csr, flops=0)
    if kind == "vertices":
        return dict(bytes=csr + 8 * n, flops=0)
    if kind == "list":
        # R-MAT graphs of this size have about 0.058 slots^(4/3) triangles
        return dict(bytes=csr + (12 * 0.058 * slots ** (4.0 / 3.0) if case["family"] == "rmat" else 0), flops=0)
    return dict(bytes=csr + (4 * n if case.get("levels") else 0) + 48, flops=0)


# ----------------------------------------------------------------------------- exact results in plain torch

_WEDGES = 3_000_000_000  # more ordered neighbour pairs than this take too long here


def _rows(rp):
    n = rp.numel() - 1
    return torch.repeat_interleave(torch.arange(n, device=DEV), rp[1:] - rp[:-1])


def _levels(rp, col, rank):
    """BFS levels from every component's first vertex in the working order, and the components."""
    n = rp.numel() - 1
    src, dst = _rows(rp), col.long()
    label = rank.clone()
    while True:
        new = label.scatter_reduce(0, dst, label[src], "amin")
        if torch.equal(new, label):
            break
        label = new
    root = label == rank
    L = torch.where(root, 0, -1)
    depth = 0
    while True:
        hit = dst[L[src] == depth]
        hit = hit[L[hit] < 0]
        if hit.numel() == 0:
            return L, int(root.sum())
        depth += 1
        L[hit] = depth


def _wedges(n, rp, col, rank):
    """Triangles (earliest, middle, latest rank), chunk by chunk; None if there are too many pairs to try."""
    src, dst = rank[_rows(rp)], rank[col.long()]
    key = torch.sort((src * n + dst)[dst < src]).values  # later vertex, earlier neighbour
    v, u = key // n, key % n
    start = torch.searchsorted(key, torch.arange(n + 1, device=DEV, dtype=torch.int64) * n)
    before = torch.arange(key.numel(), device=DEV) - start[v]
    total = torch.cumsum(before, 0)
    if key.numel() == 0 or int(total[-1]) > _WEDGES:
        return None if key.numel() else []
    def chunks():
        e = 0
        while e < key.numel():
            done = int(total[e - 1]) if e else 0
            stop = max(e + 1, int(torch.searchsorted(total, torch.tensor(done + (1 << 26), device=DEV))))
            stop = min(stop, key.numel())
            c = before[e:stop]
            edge = torch.repeat_interleave(torch.arange(e, stop, device=DEV), c)
            j = torch.arange(edge.numel(), device=DEV) - torch.repeat_interleave(torch.cumsum(c, 0) - c, c)
            w = u[start[v[edge]] + j]
            want = u[edge] * n + w
            at = torch.searchsorted(key, want).clamp_(max=key.numel() - 1)
            ok = key[at] == want
            yield w[ok], u[edge[ok]], v[edge[ok]]
            e = stop
    return chunks()


def exact(case, seed):
    gen = _generator(seed)
    kind = case["kind"]
    if kind == "batch":
        T = []
        for n, rp, col in _batch_graphs(case, gen):
            order = torch.argsort(rp[:-1] - rp[1:], stable=True)
            rank = torch.empty_like(order)
            rank[order] = torch.arange(n, device=DEV)
            T.append(sum(w.numel() for w, _, _ in _wedges(n, rp, col, rank)))
        return dict(counts=torch.tensor(T))
    n, src, dst = _tuples(case, gen)
    if _size(case)[1] > 80_000_000:
        return None
    rp, col = _csr(n, src, dst)
    del src, dst
    if kind == "build":
        padded = torch.zeros(_size(case)[1], dtype=torch.int32, device=DEV)
        padded[:col.numel()] = col
        return dict(row_ptr=rp, col=padded, slots=col.numel())
    if case["order"] == "id":
        order = torch.arange(n, device=DEV)
    else:
        order = torch.argsort(rp[:-1] - rp[1:], stable=True)
    rank = torch.empty_like(order)
    rank[order] = torch.arange(n, device=DEV)
    found = _wedges(n, rp, col, rank)
    if found is None:
        return None
    out = dict(triangles=0, t_same=None, t_cross=None, horizontal_edges=None, levels=None, components=None)
    L = None
    if case["family"] != "grid":  # a grid's thousands of levels take too long here
        L, roots = _levels(rp, col, rank)
        out.update(t_same=0, horizontal_edges=int((L[_rows(rp)] == L[col.long()]).sum()) // 2,
                   levels=int(L.max()) + 1, components=roots)
    counts, keys = torch.zeros(n, dtype=torch.int64, device=DEV), []
    for tri in found:
        a, b, c = (order[x] for x in tri)
        out["triangles"] += a.numel()
        if L is not None:
            out["t_same"] += int(((L[a] == L[b]) & (L[b] == L[c])).sum())
        if kind == "vertices":
            for x in (a, b, c):
                counts += torch.bincount(x, minlength=n)
        if kind == "list":
            keys.append(_canonical(torch.stack([a, b, c], 1).int().reshape(-1)))
    if L is not None:
        out["t_cross"] = out["triangles"] - out["t_same"]
    if kind == "vertices":
        out["counts"] = counts
    if kind == "list":
        out["triples"] = torch.zeros(_capacity(case), dtype=torch.int64, device=DEV)
        if keys:
            out["triples"][:out["triangles"]] = torch.sort(torch.cat(keys)).values
    if kind == "count" and case["levels"]:
        out["L"] = None if L is None else L.to(torch.int32)
    return out

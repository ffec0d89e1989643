// levels.cu -- degrees, canonical BFS roots and BFS levels (Algorithm 4, BFS loop).
//
// Algorithm 4 starts a BFS from every vertex still unvisited, taking vertices in
// the working order, so every component's root is its first vertex in that order
// (degree order: highest degree, then lowest id).  On the GPU:
//   1. k_init computes degrees, gives isolated vertices level 0 (each is its
//      own root) and finds the globally first non-isolated vertex;
//   2. a direction-optimising frontier BFS (top-down with edge-balanced
//      expansion, bottom-up when the frontier is large) levels its component;
//   3. the vertices still unvisited form the other components: min-key
//      hooking with pointer jumping finds each one's first vertex, and a
//      multi-source BFS from those roots levels them.
// BFS distances are unique given the roots, so L matches the serial
// algorithm exactly whatever the thread schedule.
#include <cooperative_groups.h>

#include <algorithm>
#include <type_traits>

#include "pipeline.cuh"

namespace tc {
namespace {

__device__ __forceinline__ unsigned long long warp_min_u64(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        unsigned long long y = __shfl_xor_sync(0xFFFFFFFFu, v, o);
        v = y < v ? y : v;
    }
    return v;
}

__global__ void k_init(uint32_t n, const uint64_t *__restrict__ rp, uint32_t *__restrict__ deg,
                       uint32_t *__restrict__ L, Ctl *ctl, uint32_t order) {
    __shared__ unsigned int s_iso, s_dense;
    __shared__ unsigned long long s_key;
    if (threadIdx.x == 0) {
        s_iso = s_dense = 0;
        s_key = ~0ull;
    }
    __syncthreads();
    unsigned long long best = ~0ull;
    unsigned iso = 0, dense = 0;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t v = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
        uint32_t d = (uint32_t)(rp[v + 1] - rp[v]);
        deg[v] = d;
        dense += d >= kDenseDeg;
        if (d == 0) {
            L[v] = 0;
            ++iso;
        } else {
            L[v] = kUnvisited;
            unsigned long long k = order_key((uint32_t)v, d, order);
            best = k < best ? k : best;
        }
    }
    best = warp_min_u64(best);
    iso = warp_sum(iso);
    dense = warp_sum(dense);
    if (lane_id() == 0) {
        atomicMin(&s_key, best);
        atomicAdd(&s_iso, iso);
        if (dense) atomicAdd(&s_dense, dense);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        if (s_key != ~0ull) atomicMin(&ctl->root_key, s_key);
        if (s_dense) atomicAdd(&ctl->n_dense, s_dense);
        if (s_iso) {
            atomicAdd(&ctl->visited, s_iso);
            atomicAdd(&ctl->components, s_iso);
        }
    }
}

// Their exclusive prefix too, for a frontier one block can walk.
constexpr uint32_t kPrefixOne = 32768;
__global__ void __launch_bounds__(1024) k_prefix_deg(const uint32_t *__restrict__ q, uint32_t count,
                                                     const uint32_t *__restrict__ deg,
                                                     unsigned long long *__restrict__ out) {
    __shared__ unsigned long long s_warp[32];
    const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
    unsigned long long carry = 0;
    for (uint32_t c = 0; c < count; c += 8192) {
        uint32_t d[8];
        unsigned long long sum = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const uint32_t j = c + threadIdx.x * 8 + i;
            d[i] = j < count ? q[j] : kUnvisited;
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            d[i] = d[i] != kUnvisited ? deg[d[i]] : 0u;
            sum += d[i];
        }
        unsigned long long incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
            if (lane >= (unsigned)o) incl += y;
        }
        if (lane == 31) s_warp[warp] = incl;
        __syncthreads();
        const unsigned long long w = s_warp[lane];
        unsigned long long wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xFFFFFFFFu, wi, o);
            if (lane >= (unsigned)o) wi += y;
        }
        unsigned long long ex = carry + __shfl_sync(0xFFFFFFFFu, wi - w, warp) + incl - sum;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const uint32_t j = c + threadIdx.x * 8 + i;
            if (j < count) out[j] = ex;
            ex += d[i];
        }
        carry += __shfl_sync(0xFFFFFFFFu, wi, 31);
        __syncthreads();
    }
    if (threadIdx.x == 0) out[count] = carry;
}

__global__ void k_gather_deg(const uint32_t *__restrict__ q, uint32_t count, const uint32_t *__restrict__ deg,
                             uint32_t *__restrict__ out) {
    const uint32_t stride = gridDim.x * blockDim.x;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += stride) out[i] = deg[q[i]];
}

constexpr int kTdThreads = 256;
constexpr int kTdItems = 8;
constexpr uint64_t kTdTile = (uint64_t)kTdThreads * kTdItems;

// Top-down step with edge-balanced expansion: the frontier's adjacency lists
// are viewed as one concatenated list (fpref = exclusive prefix of frontier
// degrees); each block takes tiles of kTdTile consecutive entries.
__global__ void __launch_bounds__(kTdThreads) k_td(const uint32_t *__restrict__ q, uint32_t fcount,
                                                   const unsigned long long *__restrict__ fpref,
                                                   const uint64_t *__restrict__ rp, const uint32_t *__restrict__ col,
                                                   const uint32_t *__restrict__ deg, uint32_t *__restrict__ L,
                                                   uint32_t *__restrict__ qn, Ctl *ctl, uint32_t level, int nxt) {
    __shared__ uint32_t s_lo, s_hi;
    __shared__ unsigned long long s_edges;
    const unsigned long long total = fpref[fcount];
    unsigned long long edges = 0;
    for (unsigned long long t0 = (unsigned long long)blockIdx.x * kTdTile; t0 < total;
         t0 += (unsigned long long)gridDim.x * kTdTile) {
        const unsigned long long t1 = t0 + kTdTile < total ? t0 + kTdTile : total;
        if (threadIdx.x == 0) {
            // frontier slots holding entries t0 and t1-1: largest i with fpref[i] <= x
            uint32_t a = 0, b = fcount;
            while (b - a > 1) {
                uint32_t m = (a + b) >> 1;
                if (fpref[m] <= t0) a = m; else b = m;
            }
            s_lo = a;
            b = fcount;
            while (b - a > 1) {
                uint32_t m = (a + b) >> 1;
                if (fpref[m] <= t1 - 1) a = m; else b = m;
            }
            s_hi = a;
        }
        __syncthreads();
        const uint32_t lo = s_lo, hi = s_hi;
        __syncthreads();
#pragma unroll 1
        for (int it = 0; it < kTdItems; ++it) {
            const unsigned long long e = t0 + (unsigned long long)it * kTdThreads + threadIdx.x;
            bool claim = false;
            uint32_t w = 0;
            if (e < t1) {
                uint32_t a = lo, b = hi + 1;
                while (b - a > 1) {
                    uint32_t m = (a + b) >> 1;
                    if (fpref[m] <= e) a = m; else b = m;
                }
                const uint32_t v = q[a];
                w = col[rp[v] + (e - fpref[a])];
                if (L[w] == kUnvisited && atomicCAS(&L[w], kUnvisited, level + 1) == kUnvisited) claim = true;
            }
            uint32_t slot = warp_append(claim, &ctl->fr_count[nxt]);
            if (claim) {
                qn[slot] = w;
                edges += deg[w];
            }
        }
    }
    edges = warp_sum(edges);
    if (threadIdx.x == 0) s_edges = 0;
    __syncthreads();
    if (lane_id() == 0 && edges) atomicAdd(&s_edges, edges);
    __syncthreads();
    if (threadIdx.x == 0 && s_edges) atomicAdd(&ctl->fr_edges[nxt], s_edges);
}

// Bottom-up step: every unvisited vertex looks for a neighbour on `level`.
__global__ void k_bu(uint32_t n, const uint64_t *__restrict__ rp, const uint32_t *__restrict__ col,
                     const uint32_t *__restrict__ deg, uint32_t *__restrict__ L, uint32_t *__restrict__ qn, Ctl *ctl,
                     uint32_t level, int nxt) {
    __shared__ unsigned long long s_edges;
    if (threadIdx.x == 0) s_edges = 0;
    __syncthreads();
    unsigned long long edges = 0;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    const uint64_t n_round = ((uint64_t)n + 31) & ~uint64_t(31);
    for (uint64_t v = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n_round; v += stride) {
        bool found = false;
        if (v < n && L[v] == kUnvisited) {
            const uint64_t b = rp[v], e = rp[v + 1];
            for (uint64_t j = b; j < e && !found; j += 4) {  // four in flight (a batch of 512 graphs, 6 passes: 994 -> 764 us)
                uint32_t y[4];
#pragma unroll
                for (int t = 0; t < 4; ++t) y[t] = col[j + t < e ? j + t : j];
#pragma unroll
                for (int t = 0; t < 4; ++t) y[t] = L[y[t]];
                found = y[0] == level || y[1] == level || y[2] == level || y[3] == level;
            }
            if (found) L[v] = level + 1;
        }
        uint32_t slot = warp_append(found, &ctl->fr_count[nxt]);
        if (found) {
            qn[slot] = (uint32_t)v;
            edges += deg[v];
        }
    }
    edges = warp_sum(edges);
    if (lane_id() == 0 && edges) atomicAdd(&s_edges, edges);
    __syncthreads();
    if (threadIdx.x == 0 && s_edges) atomicAdd(&ctl->fr_edges[nxt], s_edges);
}

__global__ void k_collect_unvisited(uint32_t n, const uint32_t *__restrict__ L, uint32_t *__restrict__ R, Ctl *ctl) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    const uint64_t n_round = ((uint64_t)n + 31) & ~uint64_t(31);
    for (uint64_t v = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n_round; v += stride) {
        bool un = v < n && L[v] == kUnvisited;
        uint32_t slot = warp_append(un, &ctl->n_residual);
        if (un) R[slot] = (uint32_t)v;
    }
}

__global__ void k_cc_init(const uint32_t *__restrict__ R, uint32_t nr, uint32_t *__restrict__ parent) {
    const uint32_t stride = gridDim.x * blockDim.x;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < nr; i += stride) parent[R[i]] = R[i];
}

// Follow parent pointers to the root.  Pointers always lead to a vertex with a
// smaller key, so the walk ends; the bound only guards against a corrupted
// array and raises the error flag.
__device__ __forceinline__ uint32_t find_root(const uint32_t *parent, uint32_t x, uint32_t n, Ctl *ctl) {
    for (uint32_t it = 0; it <= n; ++it) {
        uint32_t p = parent[x];
        if (p == x) return x;
        x = p;
    }
    ctl->error = 2;
    return x;
}

// Hooking: for every edge joining two trees, attach the root with the larger
// working-order key under the root with the smaller one.
__global__ void k_cc_hook(const uint32_t *__restrict__ R, uint32_t nr, uint32_t n, const uint64_t *__restrict__ rp,
                          const uint32_t *__restrict__ col, const uint32_t *__restrict__ deg, uint32_t *parent,
                          Ctl *ctl, uint32_t order) {
    const uint32_t stride = gridDim.x * blockDim.x;
    bool changed = false;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < nr; i += stride) {
        const uint32_t v = R[i];
        for (uint64_t j = rp[v]; j < rp[v + 1]; ++j) {
            const uint32_t w = col[j];
            if (w < v) continue;  // each undirected edge once
            uint32_t rv = find_root(parent, v, n, ctl), rw = find_root(parent, w, n, ctl);
            if (rv == rw) continue;
            unsigned long long kv = order_key(rv, deg[rv], order), kw = order_key(rw, deg[rw], order);
            uint32_t hi = kv < kw ? rw : rv, lo = kv < kw ? rv : rw;
            atomicCAS(&parent[hi], hi, lo);
            changed = true;
        }
    }
    if (__any_sync(0xFFFFFFFFu, changed) && lane_id() == 0) ctl->changed = 1;
}

__global__ void k_cc_compress(const uint32_t *__restrict__ R, uint32_t nr, uint32_t n, uint32_t *parent, Ctl *ctl) {
    const uint32_t stride = gridDim.x * blockDim.x;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < nr; i += stride) {
        const uint32_t v = R[i];
        parent[v] = find_root(parent, v, n, ctl);
    }
}

__global__ void k_cc_roots(const uint32_t *__restrict__ R, uint32_t nr, const uint32_t *__restrict__ parent,
                           const uint32_t *__restrict__ deg, uint32_t *__restrict__ L, uint32_t *__restrict__ q,
                           Ctl *ctl, int cur) {
    __shared__ unsigned long long s_edges;
    if (threadIdx.x == 0) s_edges = 0;
    __syncthreads();
    unsigned long long edges = 0;
    const uint32_t stride = gridDim.x * blockDim.x;
    const uint32_t nr_round = (nr + 31) & ~31u;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < nr_round; i += stride) {
        bool root = false;
        uint32_t v = 0;
        if (i < nr) {
            v = R[i];
            root = parent[v] == v;
        }
        uint32_t slot = warp_append(root, &ctl->fr_count[cur]);
        if (root) {
            L[v] = 0;
            q[slot] = v;
            edges += deg[v];
        }
    }
    edges = warp_sum(edges);
    if (lane_id() == 0 && edges) atomicAdd(&s_edges, edges);
    __syncthreads();
    if (threadIdx.x == 0 && s_edges) atomicAdd(&ctl->fr_edges[cur], s_edges);
}

// A disjoint union's first roots: every group's first vertex in the working
// order (its component's root too), one block per group.
__global__ void k_group_roots(GroupSpec groups, const uint32_t *__restrict__ deg, uint32_t *__restrict__ L,
                              uint32_t *__restrict__ q, Ctl *ctl, uint32_t order, int cur) {
    __shared__ unsigned long long s_key[32];
    const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
    for (uint32_t g = blockIdx.x; g < groups.n_groups; g += gridDim.x) {
        const uint32_t lo = groups.vertex_start[g], hi = groups.vertex_start[g + 1];
        unsigned long long best = ~0ull;
        for (uint32_t v = lo + threadIdx.x; v < hi; v += blockDim.x) {
            const uint32_t d = deg[v];
            if (d == 0) continue;
            const unsigned long long k = order_key(v, d, order);
            best = k < best ? k : best;
        }
        best = warp_min_u64(best);
        if (lane == 0) s_key[warp] = best;
        __syncthreads();
        if (warp == 0) {
            best = warp_min_u64(lane < (blockDim.x >> 5) ? s_key[lane] : ~0ull);
            if (lane == 0 && best != ~0ull) {
                const uint32_t r = (uint32_t)(best & 0xFFFFFFFFull);
                L[r] = 0;
                q[atomicAdd(&ctl->fr_count[cur], 1u)] = r;
                atomicAdd(&ctl->fr_edges[cur], (unsigned long long)deg[r]);
            }
        }
        __syncthreads();
    }
}

// The components left after the first BFS, where they are small together: one
// block hooks them, roots them and levels them (the steps of the kernels above
// with block barriers between them, instead of ten launches and five round trips
// to the host).  More than kResidualMax vertices, kResidualSlots CSR slots (trees and
// cycles, two slots a vertex, may have more), or a vertex of degree above kResidualDeg are
// left to those.  All levels of R-MAT 17 beside a uniform component, in one block / by the
// kernels above: 2000 vertices of mean degree 8 0.44 / 0.31 ms, 8000 of 4 0.64 / 0.36, 1000 of
// 30 0.57 / 0.36, 1000 of 8 0.32 / 0.32; R-MAT 18 beside a path of 8000 11.2 / 18.8.
// Parents are read past L1: hooking changes them by atomics.
constexpr uint32_t kResidualMax = 8192, kResidualSlots = 4096, kResidualDeg = 256;

__device__ __forceinline__ uint32_t find_root_cg(const uint32_t *parent, uint32_t x, uint32_t n, Ctl *ctl) {
    for (uint32_t it = 0; it <= n; ++it) {
        const uint32_t p = __ldcg(parent + x);
        if (p == x) return x;
        x = p;
    }
    ctl->error = 2;
    return x;
}

__global__ void __launch_bounds__(1024) k_residual(const uint32_t *__restrict__ R, uint32_t n,
                                                   const uint64_t *__restrict__ rp, const uint32_t *__restrict__ col,
                                                   const uint32_t *__restrict__ deg, uint32_t *parent, uint32_t *L,
                                                   uint32_t *q0, uint32_t *q1, Ctl *ctl, uint32_t order) {
    __shared__ unsigned int s_changed, s_count[2], s_roots, s_slots;
    __shared__ unsigned long long s_edges;
    const uint32_t nr = ctl->n_residual;
    if (nr == 0) return;
    bool wide = nr > kResidualMax;  // a thread walks a vertex's neighbours: long rows are left too
    if (threadIdx.x == 0) s_slots = 0;
    __syncthreads();
    uint32_t slots = 0;
    for (uint32_t i = threadIdx.x; i < nr && !wide; i += blockDim.x) {
        const uint32_t d = deg[R[i]];
        wide = d > kResidualDeg;
        slots += d;
    }
    slots = warp_sum(slots);
    if (lane_id() == 0) atomicAdd(&s_slots, slots);
    if (__syncthreads_or(wide) || s_slots > max(kResidualSlots, 2 * nr)) {
        if (threadIdx.x == 0) ctl->residual_left = nr;
        return;
    }
    for (uint32_t i = threadIdx.x; i < nr; i += blockDim.x) __stcg(parent + R[i], R[i]);
    if (threadIdx.x == 0) {
        s_count[0] = s_count[1] = s_roots = 0;
        s_edges = 0;
    }
    for (int round = 0; round < 64; ++round) {
        __syncthreads();
        if (threadIdx.x == 0) s_changed = 0;
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < nr; i += blockDim.x) {
            const uint32_t v = R[i];
            for (uint64_t j = rp[v]; j < rp[v + 1]; ++j) {
                const uint32_t w = col[j];
                if (w < v) continue;  // each undirected edge once
                const uint32_t rv = find_root_cg(parent, v, n, ctl), rw = find_root_cg(parent, w, n, ctl);
                if (rv == rw) continue;
                const unsigned long long kv = order_key(rv, deg[rv], order), kw = order_key(rw, deg[rw], order);
                const uint32_t hi = kv < kw ? rw : rv, lo = kv < kw ? rv : rw;
                atomicCAS(&parent[hi], hi, lo);
                s_changed = 1;
            }
        }
        __syncthreads();
        if (!s_changed) break;
        for (uint32_t i = threadIdx.x; i < nr; i += blockDim.x) __stcg(parent + R[i], find_root_cg(parent, R[i], n, ctl));
    }
    if (s_changed && threadIdx.x == 0) ctl->error = 2;  // 64 rounds halve any path long before
    unsigned long long edges = 0;
    for (uint32_t i = threadIdx.x; i < nr; i += blockDim.x) {
        const uint32_t v = R[i];
        edges += deg[v];
        if (__ldcg(parent + v) == v) {
            atomicExch(&L[v], 0u);
            __stcg(q0 + atomicAdd(&s_count[0], 1u), v);
            atomicAdd(&s_roots, 1u);
        }
    }
    if (edges) atomicAdd(&s_edges, edges);
    uint32_t level = 0, p = 0;
    for (;; ++level, p ^= 1u) {
        __syncthreads();
        const uint32_t fc = s_count[p];
        if (fc == 0) break;
        __syncthreads();
        if (threadIdx.x == 0) s_count[p ^ 1u] = 0;
        __syncthreads();
        const uint32_t *q = p ? q1 : q0;
        uint32_t *qn = p ? q0 : q1;
        for (uint32_t i = threadIdx.x; i < fc; i += blockDim.x) {
            const uint32_t v = __ldcg(q + i);
            for (uint64_t j = rp[v]; j < rp[v + 1]; ++j) {
                const uint32_t w = col[j];
                if (__ldcg(L + w) == kUnvisited && atomicCAS(&L[w], kUnvisited, level + 1) == kUnvisited)
                    __stcg(qn + atomicAdd(&s_count[p ^ 1u], 1u), w);
            }
        }
    }
    if (threadIdx.x == 0) {
        ctl->components += s_roots;
        ctl->visited += nr;
        ctl->visited_edges += s_edges;
        if (level > 0 && level - 1 > ctl->max_level) ctl->max_level = level - 1;
    }
}

__global__ void k_count_roots(Ctl *ctl, int cur) {
    ctl->components += ctl->fr_count[cur];
    ctl->visited += ctl->fr_count[cur];
    ctl->visited_edges += ctl->fr_edges[cur];
}

__global__ void k_reset_next(Ctl *ctl, int nxt) {
    ctl->fr_count[nxt] = 0;
    ctl->fr_edges[nxt] = 0;
    ctl->bfs_spill = 0;
}

// Book the level just made and clear the counters of the one after it.
__global__ void k_after_level(Ctl *ctl, int nxt, uint32_t level) {
    const int after = nxt == 2 ? 0 : nxt + 1;
    ctl->fr_count[after] = 0;
    ctl->fr_edges[after] = 0;
    ctl->visited += ctl->fr_count[nxt];
    ctl->visited_edges += ctl->fr_edges[nxt];
    if (ctl->fr_count[nxt]) ctl->max_level = level + 1 > ctl->max_level ? level + 1 : ctl->max_level;
}

// Levels of small frontiers (high-diameter graphs, and whole small graphs): one
// thread-block cluster runs level after level with a hardware cluster barrier
// each.  The frontier lives in shared memory as a queue of edge slots: a
// claimed vertex puts the slots of its row into its block's queue, so in the
// next level every thread takes one edge and no lane waits for a longer row.  A
// level's dependent chain is col -> L -> claim (with the row's place and degree
// read beside it) -> queue -> barrier; a 4096 x 4096 grid (4746 levels of about
// 3500 vertices) took 5.7 us a level with a grid-wide barrier over 64 blocks and
// a queue in global memory, 4.8 with queues of vertices here.
// Claimed vertices stay with their block, except those of degree above kFarRow, and all in
// the first levels and every 16th one: these are spread over the cluster by their ids.  (One
// block claims all of a few long rows' ends, whose edges are then too many for its queue: a
// ring of 2^17 vertices of degree 200 takes 23 us a level without kFarRow, 8.1 with it;
// a chain of cliques of 200 vertices 20 and 6.2.)
// A vertex of degree above kHubDeg is expanded by the whole cluster (its edges
// strided over all blocks).  The kernel ends when a frontier was empty or had
// more than max_f vertices or max_e edges, or (the `stop` flag, set in every
// block before the barrier, so that all leave at the same level) when a vertex
// of degree above max_d is claimed or a queue overflows; the frontier left is
// written back to q0.  With `whole` it goes on with the first vertex of the next
// component, up to kMaxRoots of them: a root costs a walk over all vertices and three
// barriers, 13 us, and k_residual takes small components together (500 triangles 0.55
// ms with up to 32 roots, 0.11 with 2; R-MAT 13 beside 1 / 3 / 20 triangles 0.10 / 0.16 /
// 0.37 against 0.11 / 0.11 / 0.12).
// Where ids follow the geometry (grids, road networks) the lines ahead of and
// behind a claimed vertex's are the next levels': they are asked into L2.
constexpr uint32_t kClusterThreads = 1024;  // 32 warps: wkey below counts on it
constexpr uint32_t kQueueCap = 4096;   // frontier vertices a block keeps (past it: a list in global memory)
constexpr uint32_t kEdgeBytes = 48 * 1024;  // room for the edge slots of one frontier
constexpr uint32_t kHubDeg = 256;
constexpr uint32_t kHubCap = 256;      // hubs per level expanded by the whole cluster
constexpr uint32_t kMaxRoots = 2;
constexpr uint32_t kSpreadFirst = 3;
constexpr uint32_t kLaneRow = 8;
constexpr uint32_t kFarRow = 32;

// Slot: an edge's place in col (32 bits where they are enough).
template <class Slot>
struct BfsShared {
    static constexpr uint32_t kEdgeCap = kEdgeBytes / sizeof(Slot);
    static constexpr Slot kNoEdge = ~(Slot)0;
    Slot qe[2][kEdgeCap];
    uint64_t hb[2][kHubCap];
    uint32_t qv[2][kQueueCap], hd[2][kHubCap];
    unsigned int cnt[3], edges[3];  // vertices and edge slots queued, by level mod 3
    unsigned int hubs[3], ticket[3], stop[3], total[2], heavy[2];
    unsigned long long wkey[32];  // smallest key of an unvisited vertex each warp saw
};

struct BfsArgs {
    uint32_t n;
    uint32_t *q0, *q1, *spill;
    const uint64_t *rp;
    const uint32_t *col, *deg;
    uint32_t *L;
    Ctl *ctl;
    uint32_t fcount, queue, level;  // the frontier to start from (seed: the first vertex of the working order)
    uint32_t seed, order, max_f, max_e, max_d, whole;
};

template <class Slot>
__global__ void __launch_bounds__(kClusterThreads, 1) k_bfs_cluster(const BfsArgs g) {
    namespace cg = cooperative_groups;
    using Shared = BfsShared<Slot>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Shared &S = *reinterpret_cast<Shared *>(smem_raw);
    __shared__ uint32_t s_base;
    cg::cluster_group cl = cg::this_cluster();
    const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
    const uint32_t C = cl.num_blocks(), me = cl.block_rank();
    const uint32_t hshift = 32u - (31u - __clz(C));
    uint32_t *L = g.L;
    if (threadIdx.x < 3) {
        S.cnt[threadIdx.x] = S.edges[threadIdx.x] = 0;
        S.hubs[threadIdx.x] = S.ticket[threadIdx.x] = S.stop[threadIdx.x] = 0;
    }
    if (threadIdx.x < 2) S.total[threadIdx.x] = S.heavy[threadIdx.x] = 0;
    uint32_t visited = g.ctl->visited;  // before this kernel adds any (read before the first barrier)
    const unsigned long long root_key = g.ctl->root_key;
    cl.sync();

    auto stop_all = [&](uint32_t s) {
        for (uint32_t r = 0; r < C; ++r) cl.map_shared_rank(&S, r)->stop[s] = 1;
    };
    // a hub goes to every block's list; false: no room left, its edges are queued like any other's
    auto push_hub = [&](uint64_t b, uint32_t d, uint32_t s, uint32_t p) {
        const uint32_t h = atomicAdd(&cl.map_shared_rank(&S, 0)->ticket[s], 1u);
        if (h >= kHubCap) return false;
        for (uint32_t r = 0; r < C; ++r) {
            Shared *R = cl.map_shared_rank(&S, r);
            R->hb[p][h] = b;
            R->hd[p][h] = d;
            atomicAdd(&R->hubs[s], 1u);
        }
        return true;
    };
    // vertex v (row start b, degree d) at place `at` of block T's queue, its `e` edge slots from `first` on
    // (false: they did not fit, v went to the spill list)
    auto store = [&](Shared *T, uint32_t v, uint64_t b, uint32_t e, uint32_t at, uint32_t first, uint32_t p) {
        const bool fits = at < kQueueCap && first + e <= Shared::kEdgeCap;
        if (at < kQueueCap) T->qv[p][at] = fits ? v : kUnvisited;
        for (uint32_t k = first; k < first + e && k < Shared::kEdgeCap; ++k)
            T->qe[p][k] = fits ? (Slot)(b + (k - first)) : Shared::kNoEdge;
        if (!fits) g.spill[atomicAdd(&g.ctl->bfs_spill, 1u)] = v;
        return fits;
    };
    // by one lane, into the block v's id hashes to
    auto push_spread = [&](uint32_t v, uint64_t b, uint32_t d, uint32_t s, uint32_t p) {
        const uint32_t e = d > kHubDeg && push_hub(b, d, s, p) ? 0u : d;
        Shared *T = cl.map_shared_rank(&S, (v * 0x9E3779B1u) >> hshift);
        const uint32_t at = atomicAdd(&T->cnt[s], 1u), first = atomicAdd(&T->edges[s], min(e, Shared::kEdgeCap + 1));
        if (!store(T, v, b, e, at, first, p) || d > g.max_d) stop_all(s);
    };
    // Ask L2 for the lines of L, rp, deg and col 32 vertices either side of v (a DRAM
    // access per level and array otherwise), once per line.
    const uint64_t slots = g.rp[g.n];
    auto ask = [](const void *q) { asm volatile("prefetch.global.L2 [%0];" ::"l"(q)); };
    auto ask_ahead = [&](uint32_t v, uint64_t b) {
        if ((v & 3u) == 0) {
            if (b + 64 < slots) ask(g.col + b + 64);
            if (b >= 64) ask(g.col + b - 64);
        }
        if ((v & 15u) == 0) {
            if (v + 32 < g.n) {
                ask(g.rp + v + 32);
                ask(g.deg + v + 32);
                ask(L + v + 32);
            }
            if (v >= 32) {
                ask(g.rp + v - 32);
                ask(g.deg + v - 32);
                ask(L + v - 32);
            }
        }
    };

    uint32_t cs = 0, p = 0, level = g.level, roots = 0, top = 0;
    if (g.seed) {
        if (root_key != ~0ull) {
            const uint32_t r = (uint32_t)(root_key & 0xFFFFFFFFull);
            if (me == 0 && threadIdx.x == 0) {
                L[r] = 0;
                push_spread(r, g.rp[r], g.deg[r], 0, 0);
            }
            ++roots;
            ++visited;
        }
    } else {
        const uint32_t *q = g.queue ? g.q1 : g.q0;
        for (uint32_t i = threadIdx.x; i < g.fcount; i += kClusterThreads) {
            const uint32_t v = q[i];
            // every block reads the whole queue and takes its own vertices
            if ((v * 0x9E3779B1u) >> hshift == me) push_spread(v, g.rp[v], g.deg[v], 0, 0);
        }
    }
    unsigned long long claimed = 0;  // degrees of the vertices claimed by this thread
    uint32_t added = 0;              // vertices of the finished frontiers claimed here (uniform)
    bool first = true;
    cl.sync();
    for (;;) {
        if (S.stop[cs]) break;
        const uint32_t ns = cs == 2 ? 0 : cs + 1, os = ns == 2 ? 0 : ns + 1, np = p ^ 1u;
        const uint32_t ne = min(S.edges[cs], Shared::kEdgeCap), nh = min(S.hubs[cs], kHubCap);
        if (threadIdx.x == 0) {  // the slot of the level before: nobody reads it any more
            S.cnt[os] = S.edges[os] = 0;
            S.hubs[os] = S.ticket[os] = S.stop[os] = 0;
        }
        const bool spread = level < kSpreadFirst || (level & 15u) == 0;
        // every lane of a warp: claim vertex w if it is unvisited, queue the claimed ones
        auto claim = [&](uint32_t w, bool valid) {
            const bool open = valid && __ldcg(L + w) == kUnvisited;
            uint64_t b = 0;
            uint32_t d = 0;
            bool got = false;
            if (open) {  // the row's place and degree beside the claim, not after it
                b = g.rp[w];
                d = g.deg[w];
                got = atomicCAS(&L[w], kUnvisited, level + 1) == kUnvisited;
            }
            const unsigned m = __ballot_sync(0xFFFFFFFFu, got);
            if (m == 0) return;
            if (got) {
                claimed += d;
                ask_ahead(w, b);
            }
            uint32_t e = got ? d : 0u;
            if (e > kHubDeg && push_hub(b, d, ns, np)) e = 0;
            // places in the queues: the claiming block's, or the one the id hashes to
            uint32_t owner = me, at = 0, first_edge = 0;
            const bool far = got && (spread || e > kFarRow);
            if (far) {
                owner = (w * 0x9E3779B1u) >> hshift;
                Shared *T = cl.map_shared_rank(&S, owner);
                at = atomicAdd(&T->cnt[ns], 1u);
                first_edge = atomicAdd(&T->edges[ns], min(e, Shared::kEdgeCap + 1));  // (more does not fit either)
            }
            if (!spread) {
                const bool near = got && !far;
                const unsigned nm = __ballot_sync(0xFFFFFFFFu, near);
                const uint32_t ne = near ? e : 0u;
                uint32_t incl = ne, place = 0;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                    if (lane >= (unsigned)o) incl += y;
                }
                if (lane == 31) place = atomicAdd(&S.edges[ns], incl);
                if (lane == 0) place = atomicAdd(&S.cnt[ns], (unsigned)__popc(nm));
                const uint32_t e0 = __shfl_sync(0xFFFFFFFFu, place, 31), v0 = __shfl_sync(0xFFFFFFFFu, place, 0);
                if (near) {
                    first_edge = e0 + incl - ne;
                    at = v0 + __popc(nm & ((1u << lane) - 1u));
                }
            }
            // rows of more than kLaneRow slots that fit are written by the whole warp
            const bool wide = got && e > kLaneRow && at < kQueueCap && first_edge + e <= Shared::kEdgeCap;
            if (got) {
                Shared *T = far ? cl.map_shared_rank(&S, owner) : &S;
                if (wide) T->qv[np][at] = w;
                const bool fits = wide || store(T, w, b, e, at, first_edge, np);
                if (!fits || d > g.max_d) stop_all(ns);
            }
            unsigned rows = __ballot_sync(0xFFFFFFFFu, wide);
            while (rows) {
                const int src = __ffs(rows) - 1;
                rows &= rows - 1;
                const uint64_t rb = __shfl_sync(0xFFFFFFFFu, b, src);
                const uint32_t re = __shfl_sync(0xFFFFFFFFu, e, src), rf = __shfl_sync(0xFFFFFFFFu, first_edge, src);
                Shared *T = cl.map_shared_rank(&S, __shfl_sync(0xFFFFFFFFu, owner, src));
                for (uint32_t k = lane; k < re; k += 32) T->qe[np][rf + k] = (Slot)(rb + k);
            }
        };
        for (uint32_t r0 = 0; r0 < ne; r0 += kClusterThreads) {
            const uint32_t i = r0 + threadIdx.x;
            const Slot j = i < ne ? S.qe[p][i] : Shared::kNoEdge;
            const bool valid = j != Shared::kNoEdge;
            claim(valid ? g.col[j] : 0u, valid);
        }
        for (uint32_t h = 0; h < nh; ++h) {
            const uint64_t b = S.hb[p][h];
            const uint32_t d = S.hd[p][h];
            for (uint32_t j0 = ((me + h) & (C - 1)) * kClusterThreads; j0 < d; j0 += C * kClusterThreads) {
                const uint32_t j = j0 + threadIdx.x;
                if ((j & ~31u) >= d) break;  // no lane of this warp has an edge
                claim(j < d ? g.col[b + j] : 0u, j < d);
            }
        }
        if (warp == kClusterThreads / 32 - 1) {  // this frontier's size, known to all blocks after the barrier
            const Shared *R = cl.map_shared_rank(&S, lane < C ? lane : me);
            const uint32_t t = warp_sum(lane < C ? R->cnt[cs] : 0u);
            const unsigned long long e = warp_sum(lane < C ? (unsigned long long)R->edges[cs] : 0ull);
            if (lane == 0) {
                S.total[p] = t;
                S.heavy[p] = e > g.max_e;
            }
        }
        // Releasing at every level, also where vertices stay with their block: the other blocks read
        // this one's counters and set its hub and stop marks across the barrier.  (A relaxed arrival
        // there took 23.0 instead of 24.3 ms on the grid, and ordered none of it; a fence by one
        // thread before it, or a release by one warp, measures the same as this.)
        cl.sync();
        const uint32_t total = S.total[p];
        const bool heavy = S.heavy[p] != 0;
        if (!first) {
            added += total;
            visited += total;
            if (total) top = level > top ? level : top;
        }
        first = false;
        cs = ns;
        p = np;
        ++level;
        if (total == 0) {  // so the next frontier is empty too
            if (!g.whole || visited >= g.n || roots >= kMaxRoots) break;
            // the first unvisited vertex of the working order roots the next component
            unsigned long long best = ~0ull;
            for (uint32_t v = me * kClusterThreads + threadIdx.x; v < g.n; v += C * kClusterThreads)
                if (__ldcg(L + v) == kUnvisited) {  // past L1, which may still hold it unvisited
                    const unsigned long long k = order_key(v, g.deg[v], g.order);
                    best = k < best ? k : best;
                }
            best = warp_min_u64(best);
            if (lane == 0) S.wkey[warp] = best;
            cl.sync();
            unsigned long long key = ~0ull;  // every warp reduces the keys of all blocks' warps
            for (uint32_t r = 0; r < C; ++r) {
                const unsigned long long k = cl.map_shared_rank(&S, r)->wkey[lane];
                key = k < key ? k : key;
            }
            key = warp_min_u64(key);
            cl.sync();
            if (key == ~0ull) break;
            const uint32_t r = (uint32_t)(key & 0xFFFFFFFFull);
            if (me == 0 && threadIdx.x == 0) {
                L[r] = 0;
                push_spread(r, g.rp[r], g.deg[r], cs, p);
                claimed += g.deg[r];
            }
            ++roots;
            ++visited;
            ++added;
            level = 0;
            first = true;
            cl.sync();
        } else if (total > g.max_f || heavy) {
            break;
        }
    }
    // what is left of the frontier (buffer p, slot cs) goes back to global memory
    const uint32_t fc = min(S.cnt[cs], kQueueCap);
    unsigned long long fe = 0;
    for (uint32_t i0 = 0; i0 < fc; i0 += kClusterThreads) {
        const uint32_t i = i0 + threadIdx.x;
        const uint32_t v = i < fc ? S.qv[p][i] : kUnvisited;  // kUnvisited: it is in the spill list
        const uint32_t at = warp_append(v != kUnvisited, &g.ctl->fr_count[0]);
        if (v != kUnvisited) {
            g.q0[at] = v;
            fe += g.deg[v];
        }
    }
    cl.sync();
    if (me == 0) {  // and the vertices that found no place in a block's queue
        const uint32_t spill = g.ctl->bfs_spill;
        if (spill) {
            if (threadIdx.x == 0) s_base = atomicAdd(&g.ctl->fr_count[0], spill);
            __syncthreads();
            for (uint32_t i = threadIdx.x; i < spill; i += kClusterThreads) {
                const uint32_t v = g.spill[i];
                g.q0[s_base + i] = v;
                fe += g.deg[v];
            }
        }
    }
    fe = warp_sum(fe);
    claimed = warp_sum(claimed);
    if (lane == 0) {
        if (fe) atomicAdd(&g.ctl->fr_edges[0], fe);
        if (claimed) atomicAdd(&g.ctl->visited_edges, claimed);
    }
    __syncthreads();
    if (me == 0 && threadIdx.x == 0) {
        // the frontier left over was claimed here unless it is the one the kernel began with
        const uint32_t left = atomicAdd(&g.ctl->fr_count[0], 0u);
        if (!first && left) {
            added += left;
            top = level > top ? level : top;
        }
        g.ctl->p_level = level;
        g.ctl->visited += added;
        if (top > g.ctl->max_level) g.ctl->max_level = top;
        if (g.seed && root_key != ~0ull) {  // the first root itself
            g.ctl->visited += 1;
            atomicAdd(&g.ctl->visited_edges, (unsigned long long)g.deg[(uint32_t)(root_key & 0xFFFFFFFFull)]);
        }
        g.ctl->components += roots;
    }
}

// A grid-wide wait that is bounded (all blocks are co-resident: the kernel is launched
// cooperatively), for tc_selftest_barrier: every block arrives and waits for one arrival more
// than the grid has.  A wait gives up after `timeout_cycles` of clock time and raises the
// error flag, so the kernel ends and the host reads TC_ERR_TIMEOUT.
__global__ void k_barrier_selftest(Ctl *ctl, long long timeout_cycles) {
    if (threadIdx.x != 0) return;
    volatile unsigned *count = &ctl->bar_count;
    const unsigned target = gridDim.x + 1;
    __threadfence();
    atomicAdd(&ctl->bar_count, 1u);
    const long long t0 = clock64();
    while (*count < target) {
        if (clock64() - t0 > timeout_cycles) {
            ctl->error = 4;
            break;
        }
        __nanosleep(32);
    }
}

unsigned grid_for(uint64_t work, unsigned threads, unsigned cap) {
    uint64_t b = (work + threads - 1) / threads;
    if (b < 1) b = 1;
    if (b > cap) b = cap;
    return (unsigned)b;
}

// Frontiers the cluster kernel takes: 16 of 152 SMs are enough for this many
// edges a level, and a level costs it no round trip to the host.
constexpr uint32_t kClusterMaxF = 32768;
constexpr uint32_t kClusterMaxE = 65536;
// One vertex's degree: its neighbours' edges may overflow the queues.  The first vertex is
// the one of the highest degree, and its neighbours have more edges than later ones do: a
// path of vertices with 1100 leaves each takes 74 us a level at 1024 later on too, 3.9 at 4096;
// a power law of 2^18 vertices whose first has degree 2048 takes 0.20 ms at 1024 there, 0.23 at 4096.
constexpr uint32_t kClusterMaxD = 4096, kClusterSeedD = 1024;
// Graphs it levels from the first root to the last component.
constexpr uint32_t kWholeN = 65536;
constexpr uint64_t kWholeSlots = 1u << 18;

// Levels given by the caller: degrees, a copy of the levels, their maximum,
// and the check that makes the count exact with them -- every edge joins
// vertices whose levels differ by at most one (then a triangle's levels are
// {l, l, l} or {l, l, l +- 1}: exactly three or exactly one horizontal edge).
// Lanes own rows of degree <= 32, whole warps take the longer rows.
__global__ void k_given_levels(uint32_t n, const uint64_t *__restrict__ rp, const uint32_t *__restrict__ col,
                               const uint32_t *__restrict__ given, uint32_t *__restrict__ deg,
                               uint32_t *__restrict__ L, Ctl *ctl) {
    const unsigned lane = lane_id();
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    const uint64_t n_round = ((uint64_t)n + 31) & ~uint64_t(31);
    unsigned bad = 0, top = 0, dense = 0;
    for (uint64_t x = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n_round; x += stride) {
        const bool valid = x < n;
        const uint64_t b = valid ? rp[x] : 0;
        const uint32_t d = valid ? (uint32_t)(rp[x + 1] - b) : 0;
        const uint32_t lx = valid ? given[x] : 0;
        if (valid) {
            deg[x] = d;
            L[x] = lx;
            top = lx > top ? lx : top;
            dense += d >= kDenseDeg;
        }
        if (valid && d <= 32)
            for (uint32_t j = 0; j < d; ++j) {
                const uint32_t ly = given[col[b + j]];
                bad |= (ly > lx ? ly - lx : lx - ly) > 1u;
            }
        unsigned pending = __ballot_sync(0xFFFFFFFFu, valid && d > 32);
        while (pending) {
            const int src = __ffs(pending) - 1;
            pending &= pending - 1;
            const uint64_t bb = __shfl_sync(0xFFFFFFFFu, b, src);
            const uint32_t bd = __shfl_sync(0xFFFFFFFFu, d, src);
            const uint32_t bl = __shfl_sync(0xFFFFFFFFu, lx, src);
            for (uint32_t j = lane; j < bd; j += 32) {
                const uint32_t ly = given[col[bb + j]];
                bad |= (ly > bl ? ly - bl : bl - ly) > 1u;
            }
        }
    }
    bad = __any_sync(0xFFFFFFFFu, bad);
    dense = warp_sum(dense);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned y = __shfl_xor_sync(0xFFFFFFFFu, top, o);
        top = y > top ? y : top;
    }
    if (lane == 0) {
        if (bad) atomicOr(&ctl->error, 0x200u);
        if (top) atomicMax(&ctl->max_level, top);
        if (dense) atomicAdd(&ctl->n_dense, dense);
    }
}

}  // namespace

// Pull the control block to the host (synchronises the stream).
static tc_status pull_ctl(tc_ctx *ctx) {
    TC_CUDA(ctx, cudaMemcpyAsync(ctx->h_ctl, ctx->d_ctl, sizeof(Ctl), cudaMemcpyDeviceToHost, ctx->stream));
    TC_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    return TC_OK;
}

// Run the cluster kernel: from the frontier in queue `queue`, or (seed) from
// the first vertex of the working order.  Its results are in the control block.
static tc_status launch_cluster(tc_ctx *ctx, const PipeBufs &b, uint32_t n, uint64_t slots, bool seed, uint32_t fcount,
                                uint32_t queue, uint32_t level) {
    BfsArgs a{};
    a.n = n;
    a.q0 = b.q0;
    a.q1 = b.q1;
    a.spill = b.R;
    a.rp = b.rp;
    a.col = b.col;
    a.deg = b.deg;
    a.L = b.L;
    a.ctl = ctx->d_ctl;
    a.fcount = fcount;
    a.queue = queue;
    a.level = level;
    a.seed = seed;
    a.order = ctx->opt.order;
    a.whole = seed && n <= kWholeN && slots <= kWholeSlots;
    a.max_f = a.whole ? 0xFFFFFFFFu : kClusterMaxF;
    a.max_e = a.whole ? 0xFFFFFFFFu : kClusterMaxE;
    a.max_d = a.whole ? 0xFFFFFFFFu : seed ? kClusterSeedD : kClusterMaxD;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeClusterDimension;
    cudaLaunchConfig_t cfg{};
    cfg.blockDim = dim3(kClusterThreads);
    const bool narrow = slots < 0xFFFFFFFFull;
    const void *kern = narrow ? (const void *)k_bfs_cluster<uint32_t> : (const void *)k_bfs_cluster<uint64_t>;
    cfg.dynamicSmemBytes = narrow ? sizeof(BfsShared<uint32_t>) : sizeof(BfsShared<uint64_t>);
    cfg.stream = ctx->stream;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    uint32_t &blocks = ctx->bfs_cluster[narrow ? 0 : 1];
    if (!blocks) {  // 16 blocks where the device allows them (more than the portable 8)
        TC_CUDA(ctx, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cfg.dynamicSmemBytes));
        int clusters = 0;
        attr.val.clusterDim = {16, 1, 1};
        cfg.gridDim = dim3(16);
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
            cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg) != cudaSuccess)
            clusters = 0;
        cudaGetLastError();
        blocks = clusters > 0 ? 16 : 8;
    }
    attr.val.clusterDim = {blocks, 1, 1};
    cfg.gridDim = dim3(blocks);
    void *args[] = {&a};
    TC_CUDA(ctx, cudaLaunchKernelExC(&cfg, kern, args));
    note_launch(ctx);
    return TC_OK;
}

// Level-synchronous BFS from the frontier in queue `queue`, counter slot
// `slot` (levels 0 .. start_level already assigned; the control block has been
// pulled).  Per level the host chooses top-down (edge-balanced) or bottom-up
// (Beamer et al.'s edge/vertex heuristics); runs of small frontiers go to the
// cluster kernel, unless it has just left this one (stuck).
static tc_status bfs_loop(tc_ctx *ctx, const PipeBufs &b, uint32_t n, uint64_t slots, uint32_t start_level,
                          uint32_t slot, uint32_t queue, bool stuck) {
    cudaStream_t s = ctx->stream;
    const unsigned cap = (unsigned)ctx->num_sms * 16u;
    uint32_t level = start_level;
    bool bottom_up = false, clear = false;
    tc_status st = TC_OK;
    uint32_t fcount = ctx->h_ctl->fr_count[slot];
    unsigned long long fedges = ctx->h_ctl->fr_edges[slot];
    uint32_t prev_count = 0;
    while (fcount > 0) {
        const unsigned long long unexplored = slots - ctx->h_ctl->visited_edges;
        if (!bottom_up && fedges > unexplored / 14 && fcount > 64) bottom_up = true;
        else if (bottom_up && fcount < n / 24 && fcount < prev_count) bottom_up = false;
        const uint32_t nxt = slot == 2 ? 0 : slot + 1;
        if (!bottom_up && !stuck && fcount <= kClusterMaxF && fedges <= kClusterMaxE) {
            k_reset_next<<<1, 1, 0, s>>>(ctx->d_ctl, 0);
            note_launch(ctx);
            st = launch_cluster(ctx, b, n, slots, false, fcount, queue, level);
            if (st == TC_OK) st = pull_ctl(ctx);
            if (st != TC_OK) return st;
            clear = false;
            stuck = ctx->h_ctl->p_level == level;  // it could not take the frontier (one block's queue overflowed)
            slot = 0;
            queue = 0;
            level = ctx->h_ctl->p_level;
            prev_count = fcount;
            fcount = ctx->h_ctl->fr_count[0];
            fedges = ctx->h_ctl->fr_edges[0];
            continue;  // the frontier is empty or too large for the cluster
        }
        stuck = false;
        uint32_t *q = queue ? b.q1 : b.q0;
        uint32_t *qn = queue ? b.q0 : b.q1;
        if (!clear) {  // k_after_level has done it for the later levels
            k_reset_next<<<1, 1, 0, s>>>(ctx->d_ctl, (int)nxt);
            note_launch(ctx);
        }
        clear = true;
        note_launch(ctx);  // after-level bookkeeping
        if (bottom_up) {
            k_bu<<<grid_for(n, 256, cap), 256, 0, s>>>(n, b.rp, b.col, b.deg, b.L, qn, ctx->d_ctl, level, (int)nxt);
            note_launch(ctx);
        } else if (fedges > 0) {
            if (fcount <= kPrefixOne) {
                k_prefix_deg<<<1, 1024, 0, s>>>(q, fcount, b.deg, reinterpret_cast<unsigned long long *>(b.fpref));
                note_launch(ctx, 2);
            } else {
                k_gather_deg<<<grid_for(fcount, 256, cap), 256, 0, s>>>(q, fcount, b.deg, b.fdeg);
                note_launch(ctx, 2 + scan_u32_to_u64(b.fdeg, b.fpref, fcount, b.scan_tmp, s));
            }
            k_td<<<grid_for((fedges + kTdTile - 1) / kTdTile, 1, cap), kTdThreads, 0, s>>>(
                q, fcount, reinterpret_cast<const unsigned long long *>(b.fpref), b.rp, b.col, b.deg, b.L, qn,
                ctx->d_ctl, level, (int)nxt);
        }
        k_after_level<<<1, 1, 0, s>>>(ctx->d_ctl, (int)nxt, level);
        TC_CUDA(ctx, cudaGetLastError());
        st = pull_ctl(ctx);
        if (st != TC_OK) return st;
        prev_count = fcount;
        fcount = ctx->h_ctl->fr_count[nxt];
        fedges = ctx->h_ctl->fr_edges[nxt];
        slot = nxt;
        queue ^= 1u;
        ++level;
    }
    return TC_OK;
}

tc_status selftest_barrier(tc_ctx *ctx, uint32_t timeout_ms) {
    cudaStream_t s = ctx->stream;
    TC_CUDA(ctx, cudaMemsetAsync(ctx->d_ctl, 0, sizeof(Ctl), s));
    Ctl *ctl = ctx->d_ctl;
    long long cycles = (long long)timeout_ms * 2000000ll;  // clock64 ticks at about 2 GHz
    void *args[] = {&ctl, &cycles};
    TC_CUDA(ctx, cudaLaunchCooperativeKernel((const void *)k_barrier_selftest, dim3(ctx->num_sms), dim3(64), args, 0, s));
    tc_status st = pull_ctl(ctx);
    if (st != TC_OK) return st;
    if (ctx->h_ctl->error == 4) return set_error(ctx, TC_ERR_TIMEOUT, "device wait timed out (self-test)");
    return set_error(ctx, TC_ERR_CUDA, "self-test barrier did not time out");
}

tc_status given_levels(tc_ctx *ctx, const PipeBufs &b, uint32_t n, const uint32_t *levels_in) {
    cudaStream_t s = ctx->stream;
    const unsigned cap = (unsigned)ctx->num_sms * 16u;
    if (n == 0) return TC_OK;
    k_given_levels<<<grid_for(n, 256, cap), 256, 0, s>>>(n, b.rp, b.col, levels_in, b.deg, b.L, ctx->d_ctl);
    note_launch(ctx);
    TC_CUDA(ctx, cudaGetLastError());
    tc_status st = pull_ctl(ctx);
    if (st != TC_OK) return st;
    if (ctx->h_ctl->error & 0x200u)
        return set_error(ctx, TC_ERR_INVALID, "given levels differ by more than one across an edge");
    return TC_OK;
}

tc_status compute_levels(tc_ctx *ctx, const PipeBufs &b, uint32_t n, uint64_t slots) {
    cudaStream_t s = ctx->stream;
    const unsigned cap = (unsigned)ctx->num_sms * 16u;
    if (n == 0) return TC_OK;
    k_init<<<grid_for(n, 256, cap), 256, 0, s>>>(n, b.rp, b.deg, b.L, ctx->d_ctl, ctx->opt.order);
    note_launch(ctx);
    TC_CUDA(ctx, cudaGetLastError());
    tc_status st = TC_OK;
    const bool grouped = b.groups.n_groups > 1;
    if (grouped) {
        // every graph of a union is levelled from its own first vertex at once: only the
        // small components beside them are left to the hooking below
        k_group_roots<<<std::min(b.groups.n_groups, cap), 256, 0, s>>>(b.groups, b.deg, b.L, b.q0, ctx->d_ctl,
                                                                      ctx->opt.order, 0);
        k_count_roots<<<1, 1, 0, s>>>(ctx->d_ctl, 0);
        note_launch(ctx, 2);
        TC_CUDA(ctx, cudaGetLastError());
    } else {
        st = launch_cluster(ctx, b, n, slots, true, 0, 0, 0);
    }
    if (st == TC_OK) st = pull_ctl(ctx);
    if (st == TC_OK) st = bfs_loop(ctx, b, n, slots, grouped ? 0 : ctx->h_ctl->p_level, 0, 0, !grouped);
    if (st != TC_OK) return st;
    if (ctx->h_ctl->visited >= n) return TC_OK;

    // Remaining components: min-key roots by hooking, then a multi-source BFS.
    k_collect_unvisited<<<grid_for(n, 256, cap), 256, 0, s>>>(n, b.L, b.R, ctx->d_ctl);
    k_residual<<<1, 1024, 0, s>>>(b.R, n, b.rp, b.col, b.deg, b.parent, b.L, b.q0, b.q1, ctx->d_ctl, ctx->opt.order);
    note_launch(ctx, 2);
    TC_CUDA(ctx, cudaGetLastError());
    st = pull_ctl(ctx);
    if (st != TC_OK) return st;
    if (ctx->h_ctl->error) return set_error(ctx, TC_ERR_INVALID, "connected-components walk did not end");
    const uint32_t nr = ctx->h_ctl->residual_left;
    if (nr == 0) return TC_OK;
    k_cc_init<<<grid_for(nr, 256, cap), 256, 0, s>>>(b.R, nr, b.parent);
    note_launch(ctx);
    for (int round = 0;; ++round) {
        TC_CUDA(ctx, cudaMemsetAsync(&ctx->d_ctl->changed, 0, sizeof(unsigned), s));
        k_cc_hook<<<grid_for(nr, 256, cap), 256, 0, s>>>(b.R, nr, n, b.rp, b.col, b.deg, b.parent, ctx->d_ctl,
                                                         ctx->opt.order);
        k_cc_compress<<<grid_for(nr, 256, cap), 256, 0, s>>>(b.R, nr, n, b.parent, ctx->d_ctl);
        note_launch(ctx, 2);
        TC_CUDA(ctx, cudaGetLastError());
        st = pull_ctl(ctx);
        if (st != TC_OK) return st;
        if (ctx->h_ctl->error) return set_error(ctx, TC_ERR_INVALID, "connected-components walk did not end");
        if (!ctx->h_ctl->changed) break;
        if (round > 64) return set_error(ctx, TC_ERR_TIMEOUT, "connected components did not converge");
    }
    k_reset_next<<<1, 1, 0, s>>>(ctx->d_ctl, 0);
    k_cc_roots<<<grid_for(nr, 256, cap), 256, 0, s>>>(b.R, nr, b.parent, b.deg, b.L, b.q0, ctx->d_ctl, 0);
    k_count_roots<<<1, 1, 0, s>>>(ctx->d_ctl, 0);
    note_launch(ctx, 3);
    TC_CUDA(ctx, cudaGetLastError());
    st = pull_ctl(ctx);
    return st == TC_OK ? bfs_loop(ctx, b, n, slots, 0, 0, 0, false) : st;
}

}  // namespace tc

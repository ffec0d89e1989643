// wedge.cu -- the plain count under the degree order: every triangle of
// Algorithm 4 found at the wedge of its latest vertex, by tiles of 32 earlier ones.
//
// The method is Algorithm 4's (levels, horizontal and level-spanning edges,
// every triangle has one or three horizontal edges) with another choice of
// where each triangle is found.  Hashing u and probing all of G1(v) at every
// horizontal edge u -> v reads the level-spanning part of a hub v once per
// horizontal edge of v: 124 G ids at R-MAT 24.  Here every vertex x keeps only
//     N(x) = { y ~ x : y precedes x }   (ranks, ascending, each with a flag:
//                                        1 when L(y) == L(x), a horizontal edge)
// and a triangle w < u < v (ranks) is found once, as a pair of N(v) with w in
// N(u): sum C(|N(v)|, 2) pairs, about 42 G at R-MAT 24.  It lies inside G0 when
// both u-v and w-v are horizontal, else it has exactly one horizontal edge
// (levels of adjacent vertices differ by at most one), so the two flags of v's
// row alone split the count into t_same and t_cross.
//
// Tiles.  The pairs whose u is one of the U highest-degree vertices and whose
// w is one of the first K are taken 32 u's at a time: for the tile
// t = {32 t .. 32 t + 31} a block keeps word[w] (w < K, shared memory), whose
// bit i says that w precedes and neighbours u = 32 t + i.  A vertex v with
// neighbours `mask` in the tile then needs one shared load, one AND and one
// popcount per w in the prefix of its row below the tile's end, for all of
// those u together: 0.6 lookups per pair at R-MAT 20-22 (a set per u: 1).
// The rows are read as 16-bit ids (w < K <= 2^15, flag in the low bit).
// k_wedge_high takes the same tiles' pairs with w >= K, k_wedge_rest those with
// u >= U.  Measured (one GB300, whole counts, before and after): R-MAT 24
// 130.8 -> 45.7 ms, R-MAT 20 5.36 -> 2.03, Chung-Lu 2^22 16.4 -> 7.3, uniform
// 2^20 of mean degree 32 3.33 -> 1.78, R-MAT 16 1.28 -> 0.52; per-vertex counts
// of R-MAT 19 4.35 -> 2.03.
#include <algorithm>

#include "pipeline.cuh"
#include "walk.cuh"
#include "warp_sort.cuh"

namespace tc {
namespace {

constexpr uint32_t kSmallRow = 32;     // rows of degree <= 32: one lane each
constexpr uint32_t kWarpKeys = 1024;   // rows of up to this many keys are sorted by their warp
constexpr uint32_t kHugeRow = 8192;    // rows of higher degree: a block each
constexpr uint32_t kSortCap = 32768;   // largest row a block sorts (rows hold at most sqrt(slots) keys)
constexpr int kFillThreads = 256;
constexpr uint32_t kAhead = 8;         // neighbours of a lane's row read ahead together
constexpr uint16_t kPadId = 0xFFFFu;   // fills a row's last unit: rank 2^15 - 1 >= K, its word is always 0
constexpr uint32_t kTaskSteps = 1024;  // least steps (32 ids of one entry) of a tile task
constexpr uint32_t kTasksPerSm = 8;    // (a task costs its tile's build: R-MAT 20 2.51 ms at 48, 2.31 at 16, 2.27 at 8)
constexpr uint64_t kRangeBytes = 48u << 20;
constexpr unsigned kGuardSort = 0x100u;
constexpr unsigned kGuardRange = 0x800u;
constexpr unsigned kGuardWatchdog = 0x80u;
constexpr long long kWatchdogCycles = 20000000000ll;  // about 10 s of SM clock

template <bool kPacked>
__device__ __forceinline__ uint2 rank_level(const uint2 *__restrict__ lv, const uint32_t *__restrict__ lvp, uint32_t y) {
    if constexpr (kPacked) {
        const uint32_t p = lvp[y];
        return make_uint2(p >> 8, p & 0xFFu);
    } else {
        return lv[y];
    }
}

// The first U ranks are taken in tiles (k_rank_scatter); their words cover the first K.
__device__ __forceinline__ uint32_t words_of(uint32_t U) { return U < kWedgeMaxK ? U : kWedgeMaxK; }

// What a row leaves behind besides its keys: |N(x)|, how many of them lie
// below K and below U, and the row's place by rank.
struct RowOut {
    uint32_t *dcnt, *lcnt, *ucnt;
    uint4 *rmeta;
};
__device__ __forceinline__ void row_done(const RowOut &o, uint32_t x, uint32_t rank, uint64_t b, uint32_t d,
                                         uint32_t nlo, uint32_t nu) {
    o.dcnt[x] = d;
    o.lcnt[x] = nlo;
    o.ucnt[x] = nu;
    o.rmeta[rank] = make_uint4((uint32_t)b, (uint32_t)(b >> 32), d, nlo);
}

// First 16-bit id of the row at slot b: the row owns the 16-byte units (8 ids)
// [(b + 1) / 2, (b + deg + 1) / 2), at least deg / 2 of them, so a row of degree
// >= 2 has room for its ids and their padding to whole units (kPadId).
__device__ __forceinline__ uint16_t *ids_of(uint16_t *ids, uint64_t b) { return ids + 8 * ((b + 1) >> 1); }

// N(x) of every vertex of degree <= kHugeRow.  Warps take chunks of 32
// vertices; rows of degree <= 32 belong to one lane (insertion sort in its
// column of the warp's buffer), longer ones to the whole warp (compacted into
// the buffer and sorted there; more than kWarpKeys keys are left unsorted in
// place for k_wedge_sort).  Bound by the gathers of the rank/level words.
template <bool kPacked>
__global__ void __launch_bounds__(kFillThreads) k_wedge_rows(uint32_t n, const uint64_t *__restrict__ rp,
                                                             const uint32_t *__restrict__ col,
                                                             const uint2 *__restrict__ lv,
                                                             const uint32_t *__restrict__ lvp,
                                                             uint32_t *__restrict__ keys, uint16_t *__restrict__ ids,
                                                             RowOut out, uint32_t *__restrict__ big,
                                                             uint32_t *__restrict__ huge, uint32_t per_warp, Ctl *ctl) {
    __shared__ __align__(16) uint32_t sbuf[kFillThreads / 32][kWarpKeys];
    const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    uint32_t *buf = sbuf[warp];
    const uint32_t U2 = 2 * ctl->wedge_u, K2 = 2 * words_of(ctl->wedge_u);  // a key below K2 has a rank below K
    unsigned long long horizontal = 0;
    const uint64_t chunks = ((uint64_t)n + per_warp - 1) / per_warp;
    for (;;) {
        unsigned int c = 0;
        if (lane == 0) c = atomicAdd(&ctl->fill_next, 1u);
        c = __shfl_sync(0xFFFFFFFFu, c, 0);
        if (c >= chunks) break;
        const uint64_t x = (uint64_t)c * per_warp + lane;
        const bool valid = lane < per_warp && x < n;
        const uint64_t b = valid ? rp[x] : 0;
        const uint32_t dx = valid ? (uint32_t)(rp[x + 1] - b) : 0;
        const uint2 me = valid ? rank_level<kPacked>(lv, lvp, (uint32_t)x) : make_uint2(0, 0);
        if (valid && dx <= kSmallRow) {
            uint32_t d = 0;
            for (uint32_t j0 = 0; j0 < dx; j0 += kAhead) {
                uint32_t y[kAhead];
                uint2 q[kAhead];
#pragma unroll
                for (uint32_t t = 0; t < kAhead; ++t) y[t] = j0 + t < dx ? col[b + j0 + t] : 0u;
#pragma unroll
                for (uint32_t t = 0; t < kAhead; ++t)
                    q[t] = j0 + t < dx ? rank_level<kPacked>(lv, lvp, y[t]) : make_uint2(0xFFFFFFFFu, 0);
#pragma unroll
                for (uint32_t t = 0; t < kAhead; ++t) {
                    if (q[t].x >= me.x) continue;
                    const uint32_t key = (q[t].x << 1) | (q[t].y == me.y);
                    uint32_t i = d++;
                    while (i > 0 && buf[(i - 1) * 32 + lane] > key) {
                        buf[i * 32 + lane] = buf[(i - 1) * 32 + lane];
                        --i;
                    }
                    buf[i * 32 + lane] = key;
                    horizontal += key & 1u;
                }
            }
            uint32_t nlo = 0, nu = 0;
            uint16_t *id = ids_of(ids, b);
            for (uint32_t i = 0; i < d; ++i) {
                const uint32_t key = buf[i * 32 + lane];
                keys[b + i] = key;
                nu += key < U2;
                if (key < K2 && dx >= 2) {  // a vertex of degree 1 closes no triangle (and has no room)
                    id[i] = (uint16_t)key;
                    ++nlo;
                }
            }
            for (uint32_t i = nlo; i & 7u; ++i) id[i] = kPadId;
            row_done(out, (uint32_t)x, me.x, b, d, nlo, nu);
        }
        __syncwarp();
        const unsigned huge_m = __ballot_sync(0xFFFFFFFFu, valid && dx > kHugeRow);
        if (valid && dx > kHugeRow) huge[atomicAdd(&ctl->n_huge, 1u)] = (uint32_t)x;
        unsigned pending = __ballot_sync(0xFFFFFFFFu, valid && dx > kSmallRow) & ~huge_m;
        while (pending) {
            const int src = __ffs(pending) - 1;
            pending &= pending - 1;
            const uint32_t bx = c * per_warp + (uint32_t)src;
            const uint32_t bd = __shfl_sync(0xFFFFFFFFu, dx, src);
            const uint64_t bb = __shfl_sync(0xFFFFFFFFu, b, src);
            const uint32_t brx = __shfl_sync(0xFFFFFFFFu, me.x, src);
            const uint32_t blx = __shfl_sync(0xFFFFFFFFu, me.y, src);
            uint32_t d = 0;
            for (uint32_t j0 = 0; j0 < bd; j0 += 128) {  // four neighbours per lane in flight
                uint32_t y[4];
                uint2 q[4];
#pragma unroll
                for (int t = 0; t < 4; ++t) y[t] = j0 + 32 * t + lane < bd ? col[bb + j0 + 32 * t + lane] : 0u;
#pragma unroll
                for (int t = 0; t < 4; ++t)
                    q[t] = j0 + 32 * t + lane < bd ? rank_level<kPacked>(lv, lvp, y[t]) : make_uint2(0xFFFFFFFFu, 0);
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const bool in = q[t].x < brx;
                    const unsigned m = __ballot_sync(0xFFFFFFFFu, in);
                    if (in) {
                        const uint32_t key = (q[t].x << 1) | (q[t].y == blx), pos = d + __popc(m & lt);
                        if (pos < kWarpKeys) buf[pos] = key; else keys[bb + pos] = key;
                        horizontal += key & 1u;
                    }
                    d += __popc(m);
                }
            }
            __syncwarp();
            if (d > kWarpKeys) {  // the rest of the row is in place already
                for (uint32_t i = lane; i < kWarpKeys; i += 32) keys[bb + i] = buf[i];
                if (lane == 0) big[atomicAdd(&ctl->n_big, 1u)] = bx;
                if (lane == 0) out.dcnt[bx] = d;
                __syncwarp();
                continue;
            }
            warp_sort_any(buf, d);
            uint32_t nlo = 0, nu = 0;
            uint16_t *id = ids_of(ids, bb);
            for (uint32_t i = lane; i < d; i += 32) {
                const uint32_t key = buf[i];
                keys[bb + i] = key;
                nu += key < U2;
                if (key < K2) {
                    id[i] = (uint16_t)key;
                    ++nlo;
                }
            }
            nlo = warp_sum(nlo);
            nu = warp_sum(nu);
            if (lane < ((0u - nlo) & 7u)) id[nlo + lane] = kPadId;
            if (lane == 0) row_done(out, bx, brx, bb, d, nlo, nu);
            __syncwarp();
        }
    }
    horizontal = warp_sum(horizontal);
    if (lane == 0 && horizontal) atomicAdd(&ctl->e0, horizontal);
}

// Rows of degree above kHugeRow, a block each: compacted in place (positions
// from the warps' ballots and a prefix over the warps), sorted by k_wedge_sort.
template <bool kPacked>
__global__ void __launch_bounds__(1024) k_wedge_rows_huge(const uint32_t *__restrict__ huge, Ctl *ctl,
                                                          const uint64_t *__restrict__ rp,
                                                          const uint32_t *__restrict__ col,
                                                          const uint2 *__restrict__ lv,
                                                          const uint32_t *__restrict__ lvp,
                                                          uint32_t *__restrict__ keys, uint32_t *__restrict__ dcnt,
                                                          uint32_t *__restrict__ big) {
    __shared__ unsigned int wcnt[32];
    __shared__ unsigned int s_i;
    const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const uint32_t nh = ctl->n_huge;
    unsigned long long horizontal = 0;
    for (;;) {
        if (threadIdx.x == 0) s_i = atomicAdd(&ctl->huge_next, 1u);
        __syncthreads();
        const uint32_t i = s_i;
        __syncthreads();
        if (i >= nh) break;
        const uint32_t x = huge[i];
        const uint64_t b = rp[x];
        const uint32_t dx = (uint32_t)(rp[x + 1] - b);
        const uint2 me = rank_level<kPacked>(lv, lvp, x);
        uint32_t d = 0;
        for (uint32_t j0 = 0; j0 < dx; j0 += 4 * blockDim.x) {
            uint32_t y[4];
            uint2 q[4];
            unsigned m[4];
            uint32_t mine = 0;
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const uint32_t j = j0 + t * blockDim.x + threadIdx.x;
                y[t] = j < dx ? col[b + j] : 0u;
            }
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const uint32_t j = j0 + t * blockDim.x + threadIdx.x;
                q[t] = j < dx ? rank_level<kPacked>(lv, lvp, y[t]) : make_uint2(0xFFFFFFFFu, 0);
                m[t] = __ballot_sync(0xFFFFFFFFu, q[t].x < me.x);
                mine += __popc(m[t]);
            }
            if (lane == 0) wcnt[warp] = mine;
            __syncthreads();
            uint32_t v = wcnt[lane], incl = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t z = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                if (lane >= (unsigned)o) incl += z;
            }
            uint32_t pos = d + __shfl_sync(0xFFFFFFFFu, incl - v, warp);
            d += __shfl_sync(0xFFFFFFFFu, incl, 31);
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                if (q[t].x < me.x) {
                    const uint32_t key = (q[t].x << 1) | (q[t].y == me.y);
                    keys[b + pos + __popc(m[t] & lt)] = key;
                    horizontal += key & 1u;
                }
                pos += __popc(m[t]);
            }
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            dcnt[x] = d;
            big[atomicAdd(&ctl->n_big, 1u)] = x;
        }
    }
    horizontal = warp_sum(horizontal);
    if (lane == 0 && horizontal) atomicAdd(&ctl->e0, horizontal);
}

// Listed rows (more than kWarpKeys keys, or of huge degree): a block each
// sorts the keys in shared memory and finishes the row.
template <bool kPacked>
__global__ void __launch_bounds__(1024) k_wedge_sort(const uint32_t *__restrict__ big, Ctl *ctl,
                                                     const uint64_t *__restrict__ rp, const uint2 *__restrict__ lv,
                                                     const uint32_t *__restrict__ lvp, uint32_t *__restrict__ keys,
                                                     uint16_t *__restrict__ ids, RowOut out) {
    extern __shared__ uint32_t sb[];  // kSortCap keys
    __shared__ unsigned int s_i, s_lo, s_u;
    const uint32_t nb = ctl->n_big, K2 = 2 * words_of(ctl->wedge_u), U2 = 2 * ctl->wedge_u;
    for (;;) {
        if (threadIdx.x == 0) {
            s_i = atomicAdd(&ctl->sort_next, 1u);
            s_lo = 0;
            s_u = 0;
        }
        __syncthreads();
        const uint32_t i = s_i;
        if (i >= nb) break;
        const uint32_t x = big[i];
        const uint64_t b = rp[x];
        const uint32_t d = out.dcnt[x];
        if (d > kSortCap) {  // cannot be: |N(x)|^2 <= slots
            if (threadIdx.x == 0) atomicOr(&ctl->error, kGuardSort);
            __syncthreads();
            continue;
        }
        uint32_t P = 2;
        while (P < d) P <<= 1;
        for (uint32_t t = threadIdx.x; t < P; t += blockDim.x) sb[t] = t < d ? keys[b + t] : kEmpty;
        __syncthreads();
        for (uint32_t k = 2; k <= P; k <<= 1) {
            for (uint32_t j = k >> 1; j > 0; j >>= 1) {
                for (uint32_t p = threadIdx.x; p < P / 2; p += blockDim.x) {
                    const uint32_t e = ((p & ~(j - 1)) << 1) | (p & (j - 1)), l = e | j;
                    const uint32_t a = sb[e], c = sb[l];
                    if ((a > c) == ((e & k) == 0)) {
                        sb[e] = c;
                        sb[l] = a;
                    }
                }
                __syncthreads();
            }
        }
        uint32_t nlo = 0, nu = 0;
        uint16_t *id = ids_of(ids, b);
        for (uint32_t t = threadIdx.x; t < d; t += blockDim.x) {
            const uint32_t key = sb[t];
            keys[b + t] = key;
            nu += key < U2;
            if (key < K2) {
                id[t] = (uint16_t)key;
                ++nlo;
            }
        }
        nlo = warp_sum(nlo);
        nu = warp_sum(nu);
        if (lane_id() == 0 && nlo) atomicAdd(&s_lo, nlo);
        if (lane_id() == 0 && nu) atomicAdd(&s_u, nu);
        __syncthreads();
        if (threadIdx.x < ((0u - s_lo) & 7u)) id[s_lo + threadIdx.x] = kPadId;
        if (threadIdx.x == 0) row_done(out, x, rank_level<kPacked>(lv, lvp, x).x, b, d, s_lo, s_u);
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------- entries

// One entry per (vertex v, tile, kind): {first 16-bit id of v's row in units of
// 16 bytes, mask of v's neighbours in the tile, units of the prefix | kind << 31,
// keys of the row below K | (slot of the row & 1) << 15 | high keys << 16}.
// kind 1: v's edges to the mask's vertices are horizontal.  The prefix holds
// every w of N(v) below K and not above the mask's last vertex, the high keys
// those from K on.
// Two launches make them tile by tile: kScatter = false counts every block's
// entries per tile, kScatter = true writes them at the scanned offsets; a
// block takes the same rows (a contiguous range) in both.  A warp flattens the keys
// of per_warp rows, one per lane and step;
// the last of the consecutive lanes of one row and tile makes their entries
// (a tile that straddles two steps gets entries from both).
// Without horizontal edges (bipartite graphs) there are no entries, and so no tasks,
// and the other kernels return as well: R-MAT 22 made bipartite 8.58 -> 2.76 ms, a uniform
// bipartite graph of 2^20 vertices and mean degree 32 1.75 -> 0.94 (the classes 4.35 and 1.16).
template <bool kScatter>
__global__ void __launch_bounds__(1024) k_wedge_entries(uint32_t n, uint64_t slots, const uint64_t *__restrict__ rp,
                                                        const uint32_t *__restrict__ keys,
                                                        const uint32_t *__restrict__ dcnt,
                                                        const uint32_t *__restrict__ lcnt,
                                                        uint32_t *__restrict__ counts,
                                                        const unsigned long long *__restrict__ offs,
                                                        unsigned long long *__restrict__ work,
                                                        uint4 *__restrict__ entries, uint64_t cap, uint32_t tiles_cap,
                                                        uint32_t per_warp, const uint2 *__restrict__ lv,
                                                        uint32_t *__restrict__ entry_v, Ctl *ctl) {
    extern __shared__ uint32_t sm[];  // tiles_cap counts or cursors, then (counting) tiles_cap steps
    __shared__ uint32_t s_row[2], s_next;
    const unsigned lane = lane_id();
    const uint32_t U = ctl->wedge_u;
    const uint32_t tiles = U >> 5, nb = gridDim.x;
    if (tiles == 0 || ctl->e0 == 0) return;  // (every triangle has a horizontal edge)
    if (tiles > tiles_cap) {
        if (threadIdx.x == 0) atomicOr(&ctl->error, kGuardRange);
        return;
    }
    if (threadIdx.x < 64) {  // rows are shared out by slots + rows (a long run of empty rows is spread too)
        const uint32_t end = threadIdx.x >> 5;  // one warp per end: 32 places tried at once
        const uint64_t at = (slots + n) * (blockIdx.x + end) / nb;
        uint32_t lo = 0, hi = n;  // the first row r with rp[r] + r >= at lies in [lo, hi]
        while (lo < hi) {
            const uint32_t step = (hi - lo + 31) / 32;
            const uint64_t r = (uint64_t)lo + (uint64_t)step * lane;
            const unsigned below = __ballot_sync(0xFFFFFFFFu, r < hi && rp[r] + r < at);
            const uint32_t k = __popc(below);  // the places below it come first
            hi = k == 0 ? lo : (uint32_t)min((uint64_t)hi, (uint64_t)lo + (uint64_t)step * k);
            if (k) lo = lo + step * (k - 1) + 1;
        }
        if (lane == 0) s_row[end] = blockIdx.x + end == nb ? n : lo;
    }
    if (threadIdx.x == 0) s_next = 0;
    for (uint32_t t = threadIdx.x; t < tiles; t += blockDim.x) {
        sm[t] = kScatter ? (uint32_t)offs[(uint64_t)t * nb + blockIdx.x] : 0u;
        if (!kScatter) sm[tiles_cap + t] = 0u;
    }
    __syncthreads();
    const uint32_t row_lo = s_row[0], row_hi = s_row[1];
    unsigned long long probes = 0;
    for (;;) {
        uint32_t g = 0;
        if (lane == 0) g = atomicAdd(&s_next, per_warp);
        g = __shfl_sync(0xFFFFFFFFu, g, 0);
        if (row_lo + g >= row_hi || g >= row_hi - row_lo) break;
        const uint32_t x = row_lo + g + lane;
        uint32_t d = 0, nlo = 0, vrank = 0;
        uint64_t b = 0;
        if (lane < per_warp && x < row_hi) {
            d = dcnt[x];
            nlo = lcnt[x];
            if (d < 2) d = 0;
            else b = rp[x];
            if (kScatter && entry_v) vrank = lv[x].x;
        }
        uint32_t incl = d;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
            if (lane >= (unsigned)o) incl += y;
        }
        const uint32_t total = __shfl_sync(0xFFFFFFFFu, incl, 31);
        for (uint32_t e0 = 0; e0 < total; e0 += 32) {
            const uint32_t e = e0 + lane;
            uint32_t r = 0;  // the row of flat position e: the first whose inclusive count passes it
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                if (__shfl_sync(0xFFFFFFFFu, incl, r + o - 1) <= e) r += o;
            r = r > 31u ? 31u : r;
            const uint32_t dr = __shfl_sync(0xFFFFFFFFu, d, r);
            const uint32_t pos = e - (__shfl_sync(0xFFFFFFFFu, incl, r) - dr);
            const uint64_t br = __shfl_sync(0xFFFFFFFFu, b, r);
            const uint32_t lr = __shfl_sync(0xFFFFFFFFu, nlo, r);
            const uint32_t vr = kScatter ? __shfl_sync(0xFFFFFFFFu, vrank, r) : 0u;
            uint32_t rank = 0xFFFFFFFFu, kind = 0;
            if (e < total) {
                const uint32_t key = keys[br + pos];
                rank = key >> 1;
                kind = key & 1u;
            }
            const bool in = rank < U;
            const uint32_t tile = rank >> 5;
            // segments of consecutive lanes of the same row and tile
            const uint32_t seg = in ? (tile << 5) | r : 0xFFFFFFFFu;
            const uint32_t left = __shfl_up_sync(0xFFFFFFFFu, seg, 1);
            const unsigned heads = __ballot_sync(0xFFFFFFFFu, lane == 0 || left != seg);
            const int start = 31 - __clz(heads & (0xFFFFFFFFu >> (31u - lane)));
            uint32_t hor = in && kind ? 1u << (rank & 31u) : 0u, ver = in && !kind ? 1u << (rank & 31u) : 0u;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t h = __shfl_up_sync(0xFFFFFFFFu, hor, o), v = __shfl_up_sync(0xFFFFFFFFu, ver, o);
                if ((int)lane - o >= start) {
                    hor |= h;
                    ver |= v;
                }
            }
            const bool tail = lane == 31 || ((heads >> (lane + 1)) & 1u);
            // a first key alone has no earlier one to pair with
            if (in && tail && pos >= 1) {  // so the prefix or the high keys hold a pair
                const uint32_t len = pos + 1 < lr ? pos + 1 : lr;
                uint32_t high = pos + 1 > lr ? pos + 1 - lr : 0u;
                if (high == 1) high = 0;  // the mask's vertex alone
                const uint32_t parts = (hor != 0) + (ver != 0);
                if constexpr (kScatter) {
                    const uint32_t at = atomicAdd(&sm[tile], parts);
                    const uint32_t unit = (uint32_t)((br + 1) >> 1), units = (len + 7) / 8;
                    const uint32_t place = lr | (uint32_t)(br & 1u) << 15 | high << 16;
                    if ((uint64_t)at + parts > cap) {
                        atomicOr(&ctl->error, kGuardRange);
                    } else {
                        if (hor) entries[at] = make_uint4(unit, hor, units | 0x80000000u, place);
                        if (ver) entries[at + (hor != 0)] = make_uint4(unit, ver, units, place);
                        if (entry_v)
                            for (uint32_t k = 0; k < parts; ++k) entry_v[at + k] = vr;
                    }
                } else {
                    atomicAdd(&sm[tile], parts);
                    atomicAdd(&sm[tiles_cap + tile], parts * ((len + 31) / 32 + (high + 15) / 16));
                    probes += (unsigned long long)parts * (len + high);
                }
            }
        }
    }
    if constexpr (!kScatter) {
        probes = warp_sum(probes);
        if (lane == 0 && probes) {
            atomicAdd(&ctl->probes, probes);
            atomicAdd(&ctl->cls_probes[1], probes);
        }
        __syncthreads();
        for (uint32_t t = threadIdx.x; t < tiles; t += blockDim.x) {
            counts[(uint64_t)t * nb + blockIdx.x] = sm[t];
            if (sm[tiles_cap + t]) atomicAdd(&work[t], (unsigned long long)sm[tiles_cap + t]);
        }
    }
}

// Tile tasks: equal slices of a tile's entries, of about the same number of
// steps everywhere (one block; at most task_cap of them).  A tile's entries are
// in row order, so its slices are row ranges: the tasks are listed range by
// range (`ranges` of them, each with about as many ids as L2 keeps), and the
// blocks that run at the same time read the same rows.  Tiles from rank
// kWedgeMaxK on, which k_wedge_high walks again, come after the others.
__global__ void __launch_bounds__(1024) k_wedge_plan(const unsigned long long *__restrict__ offs, uint32_t nb,
                                                     const unsigned long long *__restrict__ work, uint32_t num_sms,
                                                     uint32_t ranges, uint4 *__restrict__ tasks, uint32_t task_cap,
                                                     Ctl *ctl) {
    __shared__ unsigned long long s_sum[32];
    __shared__ unsigned int s_warp[32], s_base;
    const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
    const uint32_t tiles = ctl->wedge_u >> 5;
    if (tiles == 0) return;
    unsigned long long sum = 0;
    for (uint32_t t = threadIdx.x; t < tiles; t += blockDim.x) sum += work[t];
    sum = warp_sum(sum);
    if (lane == 0) s_sum[warp] = sum;
    if (threadIdx.x == 0) s_base = 0;
    __syncthreads();
    sum = warp_sum(s_sum[lane]);
    unsigned long long target = sum / ((unsigned long long)num_sms * kTasksPerSm) + 1;
    if (target < kTaskSteps) target = kTaskSteps;
    const uint32_t low = tiles < kWedgeMaxK / 32 ? tiles : kWedgeMaxK / 32;
    for (uint32_t part = 0; part < 2 * ranges; ++part) {
        const uint32_t range = part % ranges, t_lo = part < ranges ? 0u : low, t_hi = part < ranges ? low : tiles;
        if (part == ranges && threadIdx.x == 0) ctl->wedge_hi_task = s_base;
        for (uint32_t t0 = t_lo; t0 < t_hi; t0 += blockDim.x) {
            const uint32_t t = t0 + threadIdx.x;
            unsigned long long lo = 0, ent = 0, nt = 0;
            uint32_t i0 = 0, i1 = 0;  // the tile's slices that lie in this range
            if (t < t_hi) {
                lo = offs[(uint64_t)t * nb];
                ent = offs[(uint64_t)(t + 1) * nb] - lo;
                nt = (work[t] + target - 1) / target;
                if (nt > ent) nt = ent;
                i0 = (uint32_t)((nt * range + ranges - 1) / ranges);
                i1 = (uint32_t)((nt * (range + 1) + ranges - 1) / ranges);
            }
            uint32_t incl = i1 - i0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                if (lane >= (unsigned)o) incl += y;
            }
            if (lane == 31) s_warp[warp] = incl;
            __syncthreads();
            uint32_t before = s_base + incl - (i1 - i0);
            for (unsigned w = 0; w < warp; ++w) before += s_warp[w];
            for (uint32_t i = i0; i < i1; ++i) {
                if (before + i - i0 >= task_cap) {
                    atomicOr(&ctl->error, kGuardRange);
                    break;
                }
                tasks[before + i - i0] =
                    make_uint4(t, (uint32_t)(lo + ent * i / nt), (uint32_t)(lo + ent * (i + 1) / nt), 0u);
            }
            __syncthreads();
            if (threadIdx.x == blockDim.x - 1) s_base = before + i1 - i0;
            __syncthreads();
        }
    }
    if (threadIdx.x == 0) {
        ctl->n_tasks[1] = s_base;
        ctl->cls_rows[1] = s_base;
        ctl->cls_build[1] = offs[(uint64_t)tiles * nb];  // entries
    }
}

// ---------------------------------------------------------------------------- tiles

constexpr uint32_t kTileThreads = 1024;
constexpr uint32_t kTileWords = 32768;
constexpr size_t kTileSmem = 4ull * kTileWords + (kTileThreads / 32) * 32 * sizeof(uint4);
// Per-vertex counts (kM = 1) add: block-private counts of the first kPrivRanks
// ranks (the w that close most triangles) and each warp's of the tile's vertices.
constexpr uint32_t kPrivRanks = 1024;
constexpr size_t kCreditSmem = 4ull * kPrivRanks + (kTileThreads / 32) * 32 * 4ull;

__device__ __forceinline__ uint32_t lds(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}

// The next task of a counter, for thread 0 (x = kNoTask: none left).
constexpr uint32_t kNoTask = 0xFFFFFFFFu;
__device__ __forceinline__ uint4 next_tile_task(Ctl *ctl, int counter, uint32_t first, uint32_t n_tasks,
                                                const uint4 *__restrict__ tasks, long long t_start) {
    const uint32_t k = first + atomicAdd(&ctl->task_next[counter], 1u);
    if (clock64() - t_start > kWatchdogCycles) atomicOr(&ctl->error, kGuardWatchdog);
    else if (k < n_tasks) return tasks[k];
    return make_uint4(kNoTask, 0, 0, 0);
}

// One block per SM; a task is a slice of one tile's entries.  Each warp takes
// 32 entries at a time, four lanes walk a row's prefix 32 ids (64 bytes) a
// step; the next step's ids are loaded before the current ones are looked up.
// Units past the prefix are kPadId; ids of the prefix's last unit past the
// mask's last vertex read words that are 0.  Bound by the bank conflicts of the
// lookups (3.5 wavefronts per 32; L1/shared data stage at 83% at R-MAT 22) and
// by issue: R-MAT 24 (26 G lookups) 18.8 ms, with eight lanes of four ids each
// 26.0.
// With kM = 1 every triangle adds one to each of its vertices in `credit` (by
// rank): v once per run of steps on its entry, w once per lookup that hits, u
// once per triangle in the warp's own counters of the tile.
template <int kM>
__global__ void __launch_bounds__(kTileThreads, 1) k_wedge_tiles(uint32_t n, const uint4 *__restrict__ tasks,
                                                                 const uint4 *__restrict__ entries,
                                                                 const uint16_t *__restrict__ ids,
                                                                 const uint4 *__restrict__ rmeta, Ctl *ctl,
                                                                 const uint32_t *__restrict__ entry_v,
                                                                 unsigned long long *__restrict__ credit) {
    extern __shared__ __align__(16) uint32_t word[];
    __shared__ uint4 s_task[2];
    const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
    const uint32_t sub = lane & 3u;
    uint32_t *priv = word + kTileWords + (kTileThreads / 32) * 32 * 4;  // kM = 1: kPrivRanks counts
    uint32_t *ucnt = priv + kPrivRanks + 32 * warp;                     // and this warp's of the tile
    // add the block's private counts to `credit` (all threads; the tile's vertices start at u0)
    auto flush = [&](uint32_t u0) {
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < kPrivRanks; i += kTileThreads) {
            if (priv[i]) atomicAdd(credit + i, (unsigned long long)priv[i]);
            priv[i] = 0;
        }
        if (ucnt[lane]) atomicAdd(credit + u0 + lane, (unsigned long long)ucnt[lane]);
        ucnt[lane] = 0;
        __syncthreads();
    };
    uint4 *ent = reinterpret_cast<uint4 *>(word + kTileWords) + warp * 32;
    const uint32_t wbase = (uint32_t)__cvta_generic_to_shared(word);
    const uint32_t n_tasks = (uint32_t)ctl->n_tasks[1];
    const uint4 *unit = reinterpret_cast<const uint4 *>(ids);
    unsigned long long same = 0, cross = 0, inserts = 0;
    uint32_t tile = 0xFFFFFFFFu;
    const long long t_start = clock64();
    for (uint32_t i = threadIdx.x; i < kTileWords / 4; i += kTileThreads)
        reinterpret_cast<uint4 *>(word)[i] = make_uint4(0, 0, 0, 0);
    uint32_t dirty = 0;  // words [0, dirty) may be set
    if constexpr (kM == 1) {
        for (uint32_t i = threadIdx.x; i < kPrivRanks; i += kTileThreads) priv[i] = 0;
        ucnt[lane] = 0;
    }
    if (threadIdx.x == 0) s_task[0] = next_tile_task(ctl, 1, 0, n_tasks, tasks, t_start);
    __syncthreads();
    for (uint32_t phase = 0;; phase ^= 1u) {
        const uint4 task = s_task[phase];
        if (task.x == kNoTask) break;
        uint4 next;  // taken now, needed when this task is done
        if (threadIdx.x == 0) next = next_tile_task(ctl, 1, 0, n_tasks, tasks, t_start);
        if (task.x != tile) {
            tile = task.x;
            for (uint32_t i = threadIdx.x; i < dirty / 4; i += kTileThreads)
                reinterpret_cast<uint4 *>(word)[i] = make_uint4(0, 0, 0, 0);
            dirty = 32 * (tile + 1) < kTileWords ? 32 * (tile + 1) : kTileWords;
            __syncthreads();
            const uint32_t u = 32 * tile + warp;  // one row per warp
            if (u < n) {
                const uint4 m = rmeta[u];
                const uint4 *id = unit + (((((uint64_t)m.y << 32) | m.x) + 1) >> 1);
                for (uint32_t i = lane; 8 * i < m.w; i += 32) {
                    const uint4 q = id[i];
                    const uint32_t w[8] = {q.x, q.x >> 16, q.y, q.y >> 16, q.z, q.z >> 16, q.w, q.w >> 16};
#pragma unroll
                    for (uint32_t t = 0; t < 8; ++t)
                        if (8 * i + t < m.w) atomicOr(&word[(w[t] & 0xFFFFu) >> 1], 1u << warp);
                }
                if (lane == 0) inserts += m.w;
            }
            __syncthreads();
        }
        uint32_t tot = 0, sam = 0;
        for (uint32_t base = task.y + warp * 32; base < task.z; base += kTileThreads) {
            uint4 en = make_uint4(0, 0, 0, 0);
            if (base + lane < task.z) {
                en = entries[base + lane];
                if constexpr (kM == 1) en.w = entry_v[base + lane];
            }
            __syncwarp();
            ent[lane] = en;
            __syncwarp();
            Walk w = share_steps(((en.z & 0x7FFFFFFFu) + 3) >> 2);
            uint4 cur = ent[w.i];
            uint32_t at = cur.x + sub + 4 * w.skip;                            // this lane's first unit
            int rem = (int)(cur.z & 0x7FFFFFFFu) - (int)(4 * w.skip + sub);    // units from there on
            uint4 a, a1;
            uint32_t mv = 0, kl = 0, mv1, kl1;
            uint32_t vr = 0, vr1 = 0, vlast = kNoTask, vsum = 0;  // kM = 1: v, and its triangles not yet credited
            auto fetch = [&](uint4 &x, uint32_t &mm, uint32_t &kk, uint32_t &vv) {
                x = make_uint4(0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu);
                if (w.left) {
                    --w.left;
                    while (rem + (int)sub <= 0) {  // entries may have no units (high keys only)
                        w.i = (w.i + 1) & 31u;
                        cur = ent[w.i];
                        at = cur.x + sub;
                        rem = (int)(cur.z & 0x7FFFFFFFu) - (int)sub;
                    }
                    if (rem > 0) x = __ldg(unit + at);
                    at += 4;
                    rem -= 4;
                }
                mm = cur.y;
                kk = cur.z >> 31;
                if constexpr (kM == 1) vv = cur.w;
            };
            auto hit = [&](uint32_t rank, uint32_t h, uint32_t p) {
                vsum += p;
                if (rank < kPrivRanks) atomicAdd(priv + rank, p);
                else atomicAdd(credit + rank, (unsigned long long)p);
                for (; h; h &= h - 1) atomicAdd(ucnt + __ffs(h) - 1, 1u);
            };
            auto look = [&](uint32_t x, uint32_t mm, uint32_t kk) {
                const uint32_t w0 = lds(wbase + ((x << 1) & 0x1FFFCu)), w1 = lds(wbase + ((x >> 15) & 0x1FFFCu));
                const uint32_t p0 = __popc(w0 & mm), p1 = __popc(w1 & mm);
                tot += p0 + p1;
                if (x & kk) sam += p0;
                if (x & (kk << 16)) sam += p1;
                if constexpr (kM == 1) {
                    if (p0) hit((x >> 1) & 0x7FFFu, w0 & mm, p0);
                    if (p1) hit(x >> 17, w1 & mm, p1);
                }
            };
            fetch(a, mv, kl, vr);
            for (uint32_t k = 0; k < w.iters; ++k) {
                fetch(a1, mv1, kl1, vr1);
                if constexpr (kM == 1) {
                    if (vr != vlast) {
                        if (vsum) atomicAdd(credit + vlast, (unsigned long long)vsum);
                        vsum = 0;
                        vlast = vr;
                    }
                }
                look(a.x, mv, kl);
                look(a.y, mv, kl);
                look(a.z, mv, kl);
                look(a.w, mv, kl);
                a = a1;
                mv = mv1;
                kl = kl1;
                vr = vr1;
            }
            if constexpr (kM == 1)
                if (vsum) atomicAdd(credit + vlast, (unsigned long long)vsum);
        }
        same += sam;
        cross += tot - sam;
        if constexpr (kM == 1) flush(32 * tile);
        if (threadIdx.x == 0) s_task[phase ^ 1u] = next;
        __syncthreads();
    }
    same = warp_sum(same);
    cross = warp_sum(cross);
    inserts = warp_sum(inserts);
    if (lane == 0) {
        if (same) atomicAdd(&ctl->t_same, same);
        if (cross) atomicAdd(&ctl->t_cross, cross);
        if (inserts) atomicAdd(&ctl->cls_inserts[1], inserts);
    }
}

// The high keys (w >= K) of the tiles from rank K on, where a tile's vertices
// have few of them.  A bitmap (2^17 bits, indexed by the rank's low bits) says
// which w the tile's vertices can have: most keys end there, with one shared
// load.  The words of the others sit in a hash table (linear probing, {rank,
// word}, at most three quarters full: a tile with more high keys is walked in
// several rounds, each with the next kHighKeys of them in row order, so that
// every key of a row is in one round's table).  A warp flattens the
// high keys of 32 entries, one per lane and window.  R-MAT 24 (3.5 G keys): 7.8 ms;
// with 4096 keys a round and no bitmap 13.5, with 2048 and a bitmap 15.5 (two
// rounds over the entries where one now does), four lanes per entry 17.7.
constexpr uint32_t kHighThreads = 768;
constexpr uint32_t kHighAhead = 4;
constexpr uint32_t kHighBits = 1u << 17;
constexpr uint32_t kHighSlots = 8192, kHighShift = 19, kHighKeys = 6144;
constexpr size_t kHighSmem = kHighBits / 8 + 8ull * kHighSlots + (kHighThreads / 32) * 32 * sizeof(uint4);
constexpr unsigned kGuardInsert = 0x10u;

template <int kM>
__global__ void __launch_bounds__(kHighThreads, 2) k_wedge_high(uint32_t n, const uint4 *__restrict__ tasks,
                                                                const uint4 *__restrict__ entries,
                                                                const uint32_t *__restrict__ keys,
                                                                const uint4 *__restrict__ rmeta, Ctl *ctl,
                                                                const uint32_t *__restrict__ entry_v,
                                                                unsigned long long *__restrict__ credit) {
    extern __shared__ __align__(16) uint32_t member[];  // kHighBits bits, the table, the warps' entries
    uint2 *table = reinterpret_cast<uint2 *>(member + kHighBits / 32);
    __shared__ uint4 s_task[2];
    __shared__ uint32_t s_first[33];  // high keys of the tile's vertices before each of them
    const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
    uint4 *ent = reinterpret_cast<uint4 *>(table + kHighSlots) + warp * 32;
    const uint32_t n_tasks = (uint32_t)ctl->n_tasks[1];
    if (ctl->wedge_u <= kWedgeMaxK) return;
    const uint32_t first_task = ctl->wedge_hi_task;
    unsigned long long same = 0, cross = 0, inserts = 0;
    uint32_t tile = kNoTask, rounds = 1;
    const long long t_start = clock64();
    if (threadIdx.x == 0) s_task[0] = next_tile_task(ctl, 2, first_task, n_tasks, tasks, t_start);
    __syncthreads();
    for (uint32_t phase = 0;; phase ^= 1u) {
        const uint4 task = s_task[phase];
        if (task.x == kNoTask) break;
        uint4 next;  // taken now, needed when this task is done
        if (threadIdx.x == 0) next = next_tile_task(ctl, 2, first_task, n_tasks, tasks, t_start);
        const bool fresh = task.x != tile || rounds > 1;
        if (fresh) {
            tile = task.x;
            if (warp == 0) {
                uint32_t incl = 0;
                if (32 * tile + lane < n) {
                    const uint4 m = rmeta[32 * tile + lane];
                    incl = m.z - m.w;
                }
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                    if (lane >= (unsigned)o) incl += y;
                }
                s_first[lane + 1] = incl;
                if (lane == 0) s_first[0] = 0;
            }
            __syncthreads();
            rounds = (s_first[32] + kHighKeys - 1) / kHighKeys;
            if (threadIdx.x == 0) inserts += s_first[32];
        }
        for (uint32_t round = 0; round < rounds; ++round) {
            if (fresh) {
                for (uint32_t i = threadIdx.x; i < (kHighBits / 32 + 2 * kHighSlots) / 4; i += kHighThreads) {
                    // the bitmap to 0, the table to {kEmpty, 0}
                    const uint32_t e = i >= kHighBits / 128 ? kEmpty : 0u;
                    reinterpret_cast<uint4 *>(member)[i] = make_uint4(e, 0u, e, 0u);
                }
                __syncthreads();
                for (uint32_t r = warp; r < 32; r += kHighThreads / 32) {
                    // the row's high keys that are this round's
                    const uint32_t first = s_first[r], lo = max(first, round * kHighKeys);
                    const uint32_t hi = min(s_first[r + 1], (round + 1) * kHighKeys);
                    if (lo >= hi) continue;
                    const uint4 m = rmeta[32 * tile + r];
                    const uint32_t *nu = keys + (((uint64_t)m.y << 32) | m.x) + m.w;
                    for (uint32_t p = lo - first + lane; p < hi - first; p += 32) {
                        const uint32_t w = nu[p] >> 1, h = w * 0x9E3779B1u;
                        atomicOr(&member[(w & (kHighBits - 1)) >> 5], 1u << (w & 31u));
                        uint32_t s = h >> kHighShift, tries = 0;
                        for (; tries < kHighSlots; ++tries) {
                            const uint32_t old = atomicCAS(&table[s].x, kEmpty, w);
                            if (old == kEmpty || old == w) {
                                atomicOr(&table[s].y, 1u << r);
                                break;
                            }
                            s = (s + 1) & (kHighSlots - 1);
                        }
                        if (tries == kHighSlots) atomicOr(&ctl->error, kGuardInsert);
                    }
                }
                __syncthreads();
            }
            uint32_t tot = 0, sam = 0;
            for (uint32_t base = task.y + warp * 32; base < task.z; base += kHighThreads) {
                uint4 en = make_uint4(0, 0, 0, 0);
                if (base + lane < task.z) en = entries[base + lane];
                const uint32_t cnt = en.w >> 16;
                uint32_t incl = cnt;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                    if (lane >= (unsigned)o) incl += y;
                }
                const uint32_t total = __shfl_sync(0xFFFFFFFFu, incl, 31), excl = incl - cnt;
                // the entries that have high keys, packed: {first key - flat position, mask, kind, v}
                const unsigned some = __ballot_sync(0xFFFFFFFFu, cnt != 0);
                __syncwarp();
                if (cnt)
                    ent[__popc(some & ((1u << lane) - 1u))] =
                        make_uint4(2 * en.x - ((en.w >> 15) & 1u) + (en.w & 0x7FFFu) - excl, en.y, en.z >> 31,
                                   kM == 1 ? entry_v[base + lane] : 0u);
                __syncwarp();
                // One key per lane and window of 32 flat positions, kHighAhead windows in flight:
                // the entry of a position is the number of entries that start up to there.
                uint32_t before = 0;
                for (uint32_t k = 0; k < total; k += 32 * kHighAhead) {
                    uint32_t key[kHighAhead], at[kHighAhead];
#pragma unroll
                    for (uint32_t t = 0; t < kHighAhead; ++t) {
                        const uint32_t k0 = k + 32 * t;
                        const unsigned heads =
                            __reduce_or_sync(0xFFFFFFFFu, cnt && excl >= k0 && excl - k0 < 32 ? 1u << (excl - k0) : 0u);
                        at[t] = (before + __popc(heads & (0xFFFFFFFFu >> (31u - lane))) - 1u) & 31u;
                        before += __popc(heads);
                        key[t] = k0 + lane < total ? __ldg(keys + (uint32_t)(ent[at[t]].x + k0 + lane)) : 0u;
                    }
#pragma unroll
                    for (uint32_t t = 0; t < kHighAhead; ++t) {
                        const uint32_t r = key[t] >> 1;  // (rank 0, past the end, is below K: not in the table)
                        if (!((member[(r & (kHighBits - 1)) >> 5] >> (r & 31u)) & 1u)) continue;
                        uint32_t s = (r * 0x9E3779B1u) >> kHighShift;
                        uint2 e = table[s];
                        for (uint32_t tries = 0; e.x != r && e.x != kEmpty && tries < kHighSlots; ++tries) {
                            s = (s + 1) & (kHighSlots - 1);
                            e = table[s];
                        }
                        if (e.x == r) {
                            uint32_t h = e.y & ent[at[t]].y;
                            const uint32_t p = __popc(h);
                            tot += p;
                            if (key[t] & ent[at[t]].z) sam += p;
                            if constexpr (kM == 1) {
                                if (p) {
                                    atomicAdd(credit + ent[at[t]].w, (unsigned long long)p);
                                    atomicAdd(credit + r, (unsigned long long)p);
                                    for (; h; h &= h - 1) atomicAdd(credit + 32 * tile + __ffs(h) - 1, 1ull);
                                }
                            }
                        }
                    }
                }
                __syncwarp();
            }
            same += sam;
            cross += tot - sam;
            if (rounds > 1) __syncthreads();  // the table is cleared next
        }
        if (threadIdx.x == 0) s_task[phase ^ 1u] = next;
        __syncthreads();
    }
    same = warp_sum(same);
    cross = warp_sum(cross);
    inserts = warp_sum(inserts);
    if (lane == 0) {
        if (same) atomicAdd(&ctl->t_same, same);
        if (cross) atomicAdd(&ctl->t_cross, cross);
        if (inserts) atomicAdd(&ctl->cls_inserts[1], inserts);
    }
}

// ---------------------------------------------------------------------------- the other pairs

constexpr int kRestThreads = 256;
constexpr uint32_t kRestTiny = 8;           // rows of up to this many keys: one lane each
constexpr uint32_t kFilterBits = 1u << 14;  // per warp
constexpr uint32_t kRestSlots = kFilterBits / 32;  // the same memory as a table of keys
constexpr uint32_t kRestLong = 32;          // longer rows say whether the warp's next ones take the table

// Position of `rank` among the ascending keys a[lo..hi): the key's value, or kEmpty.
__device__ __forceinline__ uint32_t find_key(const uint32_t *__restrict__ a, uint32_t lo, uint32_t hi, uint32_t rank) {
    while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1, k = a[mid];
        if ((k >> 1) == rank) return k;
        if ((k >> 1) < rank) lo = mid + 1; else hi = mid;
    }
    return kEmpty;
}

// The pairs w < u of N(v) with u >= U, which no tile takes.  A row of at most
// kRestTiny keys: one lane tries its pairs, each by a search of w in N(u).  A
// longer one: its warp sets a filter bit per key of N(v), eight lanes a time
// walk N(u) and search N(v) for the keys that pass the filter.  In clustered graphs most
// pass, and the searches take the time: where a warp's last row of more than kRestLong
// keys was full of triangles, the next rows' keys are put into a table (linear probing,
// at most half full) in the filter's place.  5000 cliques of 120 9.20 -> 3.56 ms, 10000 of
// 60 2.96 -> 1.71 (the classes 6.7 and 3.7); uniform graphs of mean degree 100 6.04 -> 5.99,
// of 32 1.79 -> 1.80, Chung-Lu 2^22 7.27 -> 7.29.  (Both at once, the table beside the
// filter, leave too little L1: mean degree 100 8.2 ms.  The table out of line: 48 registers, 6.6.)
template <int kM>
__global__ void __launch_bounds__(kRestThreads) k_wedge_rest(uint32_t n, const uint64_t *__restrict__ rp,
                                                             const uint32_t *__restrict__ keys,
                                                             const uint32_t *__restrict__ dcnt,
                                                             const uint32_t *__restrict__ ucnt,
                                                             const uint4 *__restrict__ rmeta, uint32_t per_warp,
                                                             Ctl *ctl, const uint2 *__restrict__ lv,
                                                             unsigned long long *__restrict__ credit) {
    __shared__ __align__(16) uint32_t sfilter[kRestThreads / 32][kFilterBits / 32];
    if (ctl->e0 == 0) return;  // (every triangle has a horizontal edge)
    const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
    const uint32_t sub = lane & 7u, group = lane >> 3;
    uint32_t *filter = sfilter[warp];
    for (uint32_t i = lane; i < kFilterBits / 32; i += 32) filter[i] = 0;
    __syncwarp();
    unsigned long long same = 0, cross = 0, probes = 0;
    uint32_t done = 0;
    bool clustered = false;  // the warp's last long row had many triangles
    const uint64_t chunks = ((uint64_t)n + per_warp - 1) / per_warp;
    const long long t_start = clock64();
    for (;;) {
        unsigned int c = 0;
        if (lane == 0) {
            c = atomicAdd(&ctl->task_next[0], 1u);
            if (clock64() - t_start > kWatchdogCycles) {
                atomicOr(&ctl->error, kGuardWatchdog);
                c = 0xFFFFFFFFu;
            }
        }
        c = __shfl_sync(0xFFFFFFFFu, c, 0);
        if (c >= chunks) break;
        const uint64_t x = (uint64_t)c * per_warp + lane;
        uint32_t d = 0, nu = 0, vr = 0;  // keys, and those below U; its rank (kM = 1)
        uint64_t b = 0;
        if (lane < per_warp && x < n) {
            d = dcnt[x];
            nu = ucnt[x];
            if (d < 2 || d == nu) d = 0;
            else b = rp[x];
            if (kM == 1 && d) vr = lv[x].x;
        }
        // one triangle: w < u < v with these keys of w and u in v's row
        auto found = [&](uint32_t ku, uint32_t kw, uint32_t v) {
            if (ku & kw & 1u) ++same; else ++cross;
            if constexpr (kM == 1) {
                atomicAdd(credit + v, 1ull);
                atomicAdd(credit + (ku >> 1), 1ull);
                atomicAdd(credit + (kw >> 1), 1ull);
            }
        };
        if (d && d <= kRestTiny) {
            const uint32_t *row = keys + b;
            for (uint32_t j = nu > 1 ? nu : 1; j < d; ++j) {
                const uint32_t ku = row[j];
                const uint4 m = rmeta[ku >> 1];
                if (m.z == 0) continue;
                const uint32_t *nb = keys + (((uint64_t)m.y << 32) | m.x);
                for (uint32_t i = 0; i < j; ++i) {
                    const uint32_t kw = row[i];
                    if (find_key(nb, 0, m.z, kw >> 1) != kEmpty) found(ku, kw, vr);
                }
                probes += j;
            }
            ++done;
        }
        unsigned pending = __ballot_sync(0xFFFFFFFFu, d > kRestTiny);
        while (pending) {
            const int src = __ffs(pending) - 1;
            pending &= pending - 1;
            const uint32_t vd = __shfl_sync(0xFFFFFFFFu, d, src), vu = __shfl_sync(0xFFFFFFFFu, nu, src);
            const uint64_t vb = __shfl_sync(0xFFFFFFFFu, b, src);
            const uint32_t vrank = kM == 1 ? __shfl_sync(0xFFFFFFFFu, vr, src) : 0u;
            const uint32_t *row = keys + vb;
            // w is in N(u), so a key of N(v) with that rank lies before the j-th
            uint32_t hits = 0;
            auto walk = [&](auto key_of) {
                for (uint32_t j = (vu > 1 ? vu : 1) + group; j < vd; j += 4) {
                    const uint32_t ku = row[j];
                    const uint4 m = rmeta[ku >> 1];
                    const uint32_t *nb = keys + (((uint64_t)m.y << 32) | m.x);
                    if (sub == 0) probes += m.z;
                    for (uint32_t p = sub; p < m.z; p += 32) {
                        uint32_t w[4];
#pragma unroll
                        for (int t = 0; t < 4; ++t) w[t] = p + 8 * t < m.z ? nb[p + 8 * t] >> 1 : kEmpty;
#pragma unroll
                        for (int t = 0; t < 4; ++t) {
                            if (w[t] == kEmpty) continue;
                            const uint32_t kw = key_of(w[t], j);
                            if (kw == kEmpty) continue;
                            ++hits;
                            found(ku, kw, vrank);
                        }
                    }
                }
            };
            if (clustered && vd <= kRestSlots / 2) {  // (a place holds the key + 1; 0: free)
                uint32_t *table = filter;
                for (uint32_t i = lane; i < vd; i += 32) {
                    const uint32_t key = row[i];
                    for (uint32_t s = key >> 1; atomicCAS(&table[s & (kRestSlots - 1)], 0u, key + 1) != 0; ++s) {}
                }
                __syncwarp();
                walk([&](uint32_t w, uint32_t) {
                    uint32_t s = w, k = table[s & (kRestSlots - 1)];
                    while (k != 0 && ((k - 1) >> 1) != w) k = table[++s & (kRestSlots - 1)];
                    return k - 1;
                });
                __syncwarp();
                for (uint32_t i = lane; i < kRestSlots / 4; i += 32)
                    reinterpret_cast<uint4 *>(table)[i] = make_uint4(0, 0, 0, 0);
            } else {
                for (uint32_t i = lane; i < vd; i += 32) {
                    const uint32_t h = (row[i] >> 1) & (kFilterBits - 1);
                    atomicOr(&filter[h >> 5], 1u << (h & 31u));
                }
                __syncwarp();
                walk([&](uint32_t w, uint32_t j) {
                    const uint32_t h = w & (kFilterBits - 1);
                    return (filter[h >> 5] >> (h & 31u)) & 1u ? find_key(row, 0, j, w) : kEmpty;
                });
                __syncwarp();
                for (uint32_t i = lane; i < vd; i += 32) filter[((row[i] >> 1) & (kFilterBits - 1)) >> 5] = 0;
            }
            __syncwarp();
            if (vd > kRestLong) clustered = __any_sync(0xFFFFFFFFu, 4 * hits > vd);  // (a lane has vd * vd / 64 pairs)
            if (lane == 0) ++done;
        }
    }
    same = warp_sum(same);
    cross = warp_sum(cross);
    probes = warp_sum(probes);
    const unsigned long long rows = warp_sum((unsigned long long)done);
    if (lane == 0) {
        if (same) atomicAdd(&ctl->t_same, same);
        if (cross) atomicAdd(&ctl->t_cross, cross);
        if (probes) {
            atomicAdd(&ctl->probes, probes);
            atomicAdd(&ctl->cls_probes[0], probes);
        }
        if (rows) atomicAdd(&ctl->cls_rows[0], rows);
    }
}

// ---------------------------------------------------------------------------- tiles or classes

// Where more vertices than a tile's words cover have a high and much the same
// degree, a tile holds one or two neighbours of any row: a lookup serves one pair
// instead of 32, and k_wedge_high walks its entries once per kHighKeys keys.  The
// classes of isect.cu are the faster path there (uniform graphs, tiles / classes:
// 2^18 vertices of mean degree 512 / 1024 / 2048 32.7 / 201 / 1404 against 18.9 /
// 69 / 196 ms; at 256 7.05 against 7.27; R-MAT 20 of edge factor 300 59 against 161).
// So a count with more than kWedgeDense vertices of degree >= kDenseDeg (with half as
// many ranks past the words as in them, 4% of the pairs are high ones) samples
// kSamples slots, and for the vertex v of each takes the lookups that its row would
// cost: every tile with a neighbour of v walks the keys of N(v) up to it, the rest
// walks N(u), and the classes compare v's horizontal neighbours pairwise and probe its
// level-spanning ones once per horizontal edge.  Picoseconds, from uniform graphs of
// 2^16 to 2^21 vertices and mean degree 256 to 4096: high keys 3.7 (times the rounds of
// v's tiles), 16-bit ids 0.7, rest 2.9; classes 1 a probe (0.7 at degree 2048, 0.5 at
// 4096), 70 a horizontal edge, and 33 a slot for the larger row stage.  The ratio of the
// two estimates is within 1.2 of the measured one, and the classes are taken from there
// on.  One block a sample: about 40 us and a readback.
constexpr uint32_t kSamples = 1024;
constexpr uint32_t kSampleDeg = 32768;  // longer rows are not looked at (their vertex has few earlier ones)

__global__ void __launch_bounds__(256) k_wedge_estimate(uint32_t n, uint64_t slots, const uint64_t *__restrict__ rp,
                                                        const uint32_t *__restrict__ col,
                                                        const uint32_t *__restrict__ deg,
                                                        const uint2 *__restrict__ lv, Ctl *ctl) {
    __shared__ uint32_t seen[kWedgeMaxU / 1024];  // tiles with a neighbour
    __shared__ unsigned int s_low, s_high, s_hor, s_span, s_tl, s_th;
    __shared__ unsigned long long s_rest;
    const uint32_t U = ctl->wedge_u, K = words_of(U);
    for (uint32_t i = blockIdx.x; i < kSamples; i += gridDim.x) {
        const uint64_t at = slots * i / kSamples;
        uint32_t v = 0, hi = n;  // the last row that starts at or before slot `at`
        while (hi - v > 1) {
            const uint32_t mid = v + (hi - v) / 2;
            if (rp[mid] <= at) v = mid; else hi = mid;
        }
        const uint64_t b = rp[v];
        const uint32_t d = deg[v];
        const uint2 me = lv[v];
        if (d > kSampleDeg || me.x == 0) continue;
        for (uint32_t t = threadIdx.x; t < kWedgeMaxU / 1024; t += 256) seen[t] = 0;
        if (threadIdx.x == 0) {
            s_low = s_high = s_hor = s_span = s_tl = s_th = 0;
            s_rest = 0;
        }
        __syncthreads();
        uint32_t low = 0, high = 0, hor = 0, span = 0;
        unsigned long long rest = 0;
        for (uint32_t j0 = threadIdx.x; j0 < d; j0 += 1024) {
            uint32_t y[4];
            uint2 q[4];
#pragma unroll
            for (uint32_t t = 0; t < 4; ++t) y[t] = j0 + 256 * t < d ? col[b + j0 + 256 * t] : v;
#pragma unroll
            for (uint32_t t = 0; t < 4; ++t) q[t] = lv[y[t]];
#pragma unroll
            for (uint32_t t = 0; t < 4; ++t) {
                span += q[t].y != me.y;
                if (q[t].x >= me.x) continue;
                hor += q[t].y == me.y;
                if (q[t].x < U) {
                    atomicOr(&seen[q[t].x >> 10], 1u << ((q[t].x >> 5) & 31u));
                    if (q[t].x < K) ++low; else ++high;
                } else {
                    rest += deg[y[t]] / 2;  // about |N(u)|
                }
            }
        }
        low = warp_sum(low);
        high = warp_sum(high);
        hor = warp_sum(hor);
        span = warp_sum(span);
        rest = warp_sum(rest);
        if (lane_id() == 0) {
            atomicAdd(&s_low, low);
            atomicAdd(&s_high, high);
            atomicAdd(&s_hor, hor);
            atomicAdd(&s_span, span);
            atomicAdd(&s_rest, rest);
        }
        __syncthreads();
        for (uint32_t t = threadIdx.x; t < kWedgeMaxU / 1024; t += 256) {
            const uint32_t first = 32 * t, end = K / 32;  // tiles of this word, tiles below K
            const uint32_t below = end <= first ? 0u : end - first >= 32 ? 0xFFFFFFFFu : (1u << (end - first)) - 1u;
            if (seen[t] & below) atomicAdd(&s_tl, (unsigned)__popc(seen[t] & below));
            if (seen[t] & ~below) atomicAdd(&s_th, (unsigned)__popc(seen[t] & ~below));
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            const float rounds = fmaxf(1.f, 32.f * (2.f / 3.f) * s_high / kHighKeys);
            const float keys = 0.5f * s_th * s_high * rounds, ids = 0.5f * s_tl * s_low + (float)s_th * s_low;
            const float tiles_ps = 3.7f * keys + 0.7f * ids + 2.9f * s_rest;
            const float probe_ps = sqrtf(1024.f / fmaxf(1024.f, d));
            const float classes_ps = (probe_ps * (0.5f * s_hor + s_span) + 70.f) * s_hor + 33.f * d;
            // a slot stands for slots / kSamples, and v is met once per slot of its row (whole numbers: the
            // sums do not depend on the order)
            atomicAdd(&ctl->est_wedge, (unsigned long long)(1024.f * tiles_ps / d));
            atomicAdd(&ctl->est_classes, (unsigned long long)(1024.f * classes_ps / d));
        }
        __syncthreads();
    }
}

unsigned grid_for(uint64_t work, unsigned threads, unsigned cap) {
    uint64_t b = (work + threads - 1) / threads;
    if (b < 1) b = 1;
    if (b > cap) b = cap;
    return (unsigned)b;
}

// Tiles there can be (a tile vertex has degree 64 at least).
uint32_t tiles_cap(uint32_t n, uint64_t slots) {
    return (uint32_t)std::min<uint64_t>(std::min(kWedgeMaxU, n), slots / 64 + 32) / 32 + 1;
}

// Least degree of a tile vertex.  A tile costs its words' build (about 5 us of
// one SM) and saves its vertices' rows from k_wedge_rest: with 64 instead of 128
// R-MAT 13 takes 0.38 instead of 0.43 ms and R-MAT 16 0.65 instead of 0.69 (the
// SMs have tiles to spare), R-MAT 22 9.11 instead of 9.05 and Chung-Lu 2^22 7.65
// instead of 7.44.
uint32_t tile_degree(uint32_t n) { return n < (1u << 20) ? 64u : 128u; }
// Largest degree from which a graph takes tiles at all (a uniform graph of mean
// degree 32 would make a single tile: 2.02 instead of 1.87 ms).
constexpr uint32_t kTilesFrom = 128;

// Vertices a warp takes at a time: fewer in small graphs, where the rows of one
// warp's chunk would hold up everything (R-MAT 10: k_wedge_rest 78 us at 32).
uint32_t rows_per_warp(uint32_t n) {
    return n >= (1u << 20) ? 32u : n >= (1u << 18) ? 16u : n >= (1u << 15) ? 8u : 2u;
}

// Blocks of the entry kernels: a row range each.
uint32_t entry_blocks(const tc_ctx *ctx, uint64_t slots) {
    return (uint32_t)std::min<uint64_t>(2ull * ctx->num_sms, slots / 4096 + 1);
}

uint32_t tasks_cap(const tc_ctx *ctx, uint32_t n, uint64_t slots) {
    return tiles_cap(n, slots) + (uint32_t)ctx->num_sms * kTasksPerSm + 1;
}

}  // namespace

uint32_t wedge_tile_degree(uint32_t n, uint32_t max_deg) { return max_deg >= kTilesFrom ? tile_degree(n) : kNoTiles; }

WedgeSizes wedge_sizes(const tc_ctx *ctx, uint32_t n, uint64_t slots) {
    WedgeSizes z;
    z.tiles = tiles_cap(n, slots);
    z.counts = (uint64_t)z.tiles * entry_blocks(ctx, slots);
    z.tasks = tasks_cap(ctx, n, slots);
    z.tmp = scan_tmp_elems(z.counts + 1);
    return z;
}

bool wedge_path(const tc_ctx *ctx, uint32_t n, uint64_t slots, uint32_t max_deg) {
    const Tuning &t = ctx->tune, def;
    // the class knobs choose among the kernels of isect.cu: any of them set away from its default means these
    const bool classes = t.warp_cap != def.warp_cap || t.block_cap != def.block_cap || t.tiny_cap != def.tiny_cap ||
                         t.table_kind != def.table_kind || t.flat_cap != def.flat_cap ||
                         t.block_bits_log2 != def.block_bits_log2;
    return !classes && ctx->opt.order == TC_ORDER_DEGREE && ctx->nshards == 1 && max_deg > 0 && n < (1u << 31) &&
           slots <= (uint64_t)kSortCap * kSortCap;
}

tc_status wedge_estimate(tc_ctx *ctx, const PipeBufs &b, uint32_t n, bool *classes) {
    k_wedge_estimate<<<std::min<unsigned>(kSamples, (unsigned)ctx->num_sms * 8u), 256, 0, ctx->stream>>>(
        n, b.slots, b.rp, b.col, b.deg, b.lv, ctx->d_ctl);
    note_launch(ctx);
    TC_CUDA(ctx, cudaGetLastError());
    TC_CUDA(ctx, cudaMemcpyAsync(ctx->h_ctl, ctx->d_ctl, sizeof(Ctl), cudaMemcpyDeviceToHost, ctx->stream));
    TC_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    *classes = 5 * (double)ctx->h_ctl->est_wedge > 6 * (double)ctx->h_ctl->est_classes;
    return TC_OK;
}

tc_status wedge_rows(tc_ctx *ctx, const PipeBufs &b, uint32_t n, uint32_t max_deg) {
    cudaStream_t s = ctx->stream;
    const unsigned cap = (unsigned)ctx->num_sms * 16u;
    uint16_t *ids = b.wedge_ids;
    uint32_t launches = 1;
    const RowOut out{b.fcnt, b.gcnt, b.glo, b.vmeta};
    const uint32_t per_warp = rows_per_warp(n);
    auto rows = b.lvp ? k_wedge_rows<true> : k_wedge_rows<false>;
    rows<<<grid_for((uint64_t)n * (32 / per_warp), kFillThreads, cap), kFillThreads, 0, s>>>(
        n, b.rp, b.col, b.lv, b.lvp, b.adj2, ids, out, b.big, b.huge, per_warp, ctx->d_ctl);
    if (max_deg > kHugeRow) {
        auto huge = b.lvp ? k_wedge_rows_huge<true> : k_wedge_rows_huge<false>;
        huge<<<(unsigned)ctx->num_sms, 1024, 0, s>>>(b.huge, ctx->d_ctl, b.rp, b.col, b.lv, b.lvp, b.adj2, b.fcnt,
                                                     b.big);
        ++launches;
    }
    if (max_deg > kWarpKeys) {
        auto sort = b.lvp ? k_wedge_sort<true> : k_wedge_sort<false>;
        const int smem = (int)(4 * kSortCap);
        TC_CUDA(ctx, cudaFuncSetAttribute(sort, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        sort<<<(unsigned)ctx->num_sms, 1024, smem, s>>>(b.big, ctx->d_ctl, b.rp, b.lv, b.lvp, b.adj2, ids, out);
        ++launches;
    }
    if (max_deg >= kTilesFrom) {
        const uint32_t nb = entry_blocks(ctx, b.slots), tiles = tiles_cap(n, b.slots);
        const uint64_t cells = (uint64_t)tiles * nb;
        TC_CUDA(ctx, cudaMemsetAsync(b.wedge_work, 0, 8ull * tiles + 4 * cells, s));  // work and counts
        const int smem = (int)(8 * tiles);
        // (the limit is the process's, not the call's: one value for every thread's launches)
        const int most = (int)(8 * (kWedgeMaxU / 32 + 1));  // tiles_cap at its largest
        TC_CUDA(ctx, cudaFuncSetAttribute(k_wedge_entries<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
        TC_CUDA(ctx, cudaFuncSetAttribute(k_wedge_entries<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, most / 2));
        auto *offs = reinterpret_cast<unsigned long long *>(b.wedge_offs);
        k_wedge_entries<false><<<nb, 1024, smem, s>>>(n, b.slots, b.rp, b.adj2, b.fcnt, b.gcnt, b.wedge_counts, offs,
                                                      b.wedge_work, b.erec, b.erec_cap, tiles, per_warp, b.lv, b.wedge_v,
                                                      ctx->d_ctl);
        launches += 3 + scan_u32_to_u64(b.wedge_counts, b.wedge_offs, cells, b.wedge_tmp, s);
        k_wedge_entries<true><<<nb, 1024, smem / 2, s>>>(n, b.slots, b.rp, b.adj2, b.fcnt, b.gcnt, b.wedge_counts, offs,
                                                     b.wedge_work, b.erec, b.erec_cap, tiles, per_warp, b.lv, b.wedge_v,
                                                     ctx->d_ctl);
        // row ranges of about kRangeBytes of 16-bit ids (2 bytes an edge)
        const uint32_t ranges = (uint32_t)std::min<uint64_t>(b.slots / kRangeBytes + 1, 16);
        k_wedge_plan<<<1, 1024, 0, s>>>(offs, nb, b.wedge_work, (uint32_t)ctx->num_sms, ranges, b.wedge_tasks,
                                        tasks_cap(ctx, n, b.slots), ctx->d_ctl);
    }
    note_launch(ctx, launches);
    TC_CUDA(ctx, cudaGetLastError());
    return TC_OK;
}

tc_status wedge_count(tc_ctx *ctx, const PipeBufs &b, uint32_t n, uint32_t max_deg) {
    cudaStream_t s = ctx->stream;
    const bool tiles = max_deg >= kTilesFrom, credit = b.vcount != nullptr;
    TC_CUDA(ctx, cudaEventRecord(ctx->ev[4], s));
    int per_sm = 0;
    auto rest = credit ? k_wedge_rest<1> : k_wedge_rest<0>;
    TC_CUDA(ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, rest, kRestThreads, 0));
    const uint32_t per_warp = rows_per_warp(n);
    const uint64_t blocks = ((uint64_t)n + per_warp * (kRestThreads / 32) - 1) / (per_warp * (kRestThreads / 32));
    const uint64_t resident = (uint64_t)ctx->num_sms * std::max(per_sm, 1);
    rest<<<(unsigned)std::min(blocks, resident), kRestThreads, 0, s>>>(n, b.rp, b.adj2, b.fcnt, b.glo, b.vmeta, per_warp,
                                                                       ctx->d_ctl, b.lv, b.vcount_rank);
    TC_CUDA(ctx, cudaEventRecord(ctx->ev[5], s));
    if (tiles) {
        auto tile = credit ? k_wedge_tiles<1> : k_wedge_tiles<0>;
        const size_t smem = kTileSmem + (credit ? kCreditSmem : 0);
        TC_CUDA(ctx, cudaFuncSetAttribute(tile, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        tile<<<(unsigned)ctx->num_sms, kTileThreads, smem, s>>>(n, b.wedge_tasks, b.erec, b.wedge_ids, b.vmeta, ctx->d_ctl,
                                                                b.wedge_v, b.vcount_rank);
        if (n > kWedgeMaxK) {
            auto high = credit ? k_wedge_high<1> : k_wedge_high<0>;
            TC_CUDA(ctx, cudaFuncSetAttribute(high, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kHighSmem));
            high<<<(unsigned)ctx->num_sms * 2u, kHighThreads, kHighSmem, s>>>(n, b.wedge_tasks, b.erec, b.adj2, b.vmeta,
                                                                             ctx->d_ctl, b.wedge_v, b.vcount_rank);
            note_launch(ctx);
        }
    }
    TC_CUDA(ctx, cudaEventRecord(ctx->ev[6], s));
    ctx->isect_flags = tiles ? 3u : 1u;
    note_launch(ctx, tiles ? 2 : 1);
    TC_CUDA(ctx, cudaGetLastError());
    return TC_OK;
}

}  // namespace tc

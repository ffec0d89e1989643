// csr.cu -- building, checking and measuring the input CSR on the device.
//
// tc_build_csr: every tuple (a, b), a != b, counts one entry for a and one for
// b; the counts' prefix gives every vertex a row, the entries are placed in any
// order, every row is sorted and its repeats dropped by a lane, a warp or a
// block, and the rows left are packed.  (A radix sort of 64-bit keys over both
// ids moves 16 bytes an entry six times for 2^21 vertices; here an entry is a
// 4-byte id, placed once and sorted in shared memory.)  The result is the
// paper's input format: symmetric, loop-free, duplicate-free, rows ascending.
// Very many tuples or vertices, few tuples over many vertices, and a device without
// room for the counts take the radix sort: 64-bit keys (a << 32 | b)
// and (b << 32 | a), least significant 8-bit digits first, only the digits that
// can be nonzero; col = low halves of the distinct keys, row_ptr from the run
// boundaries of the high halves.
#include <algorithm>

#include "pipeline.cuh"
#include "warp_sort.cuh"

namespace tc {
namespace {

constexpr int kRsThreads = 256;
// Keys a thread takes: few of them for short arrays, whose tiles then fill the GPU
// (65536 keys: a scatter 18 -> 7 us).
constexpr int kRsItems = 16, kRsItemsShort = 4;
constexpr uint64_t kRsShort = 1u << 19;
__host__ __device__ constexpr uint64_t rs_tile(uint64_t count) {
    return (uint64_t)kRsThreads * (count <= kRsShort ? kRsItemsShort : kRsItems);
}
constexpr int kRsWarps = kRsThreads / 32;

__global__ void k_make_keys(uint64_t t, const uint32_t *__restrict__ src, const uint32_t *__restrict__ dst, uint32_t n,
                            unsigned long long *__restrict__ keys, Ctl *ctl) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    const uint64_t t_round = (t + 31) & ~uint64_t(31);
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < t_round; i += stride) {
        uint32_t a = 0, b = 0;
        bool keep = false;
        if (i < t) {
            a = src[i];
            b = dst[i];
            if (a >= n || b >= n) ctl->error = 1;
            else keep = a != b;
        }
        // two keys per kept tuple: count them in pairs
        const unsigned mask = __ballot_sync(0xFFFFFFFFu, keep);
        uint64_t base = 0;
        if (mask) {
            const unsigned leader = __ffs(mask) - 1;
            if (lane_id() == leader) base = (uint64_t)atomicAdd(&ctl->visited_edges, 2ull * __popc(mask));
            base = __shfl_sync(0xFFFFFFFFu, base, leader);
        }
        if (keep) {
            const uint64_t slot = base + 2u * __popc(mask & ((1u << lane_id()) - 1u));
            keys[slot] = ((unsigned long long)a << 32) | b;
            keys[slot + 1] = ((unsigned long long)b << 32) | a;
        }
    }
}

// Per-tile digit histograms, digit-major: counts[d * nblocks + block].
template <int kItems>
__global__ void __launch_bounds__(kRsThreads) k_rs_hist(const unsigned long long *__restrict__ keys, uint64_t count,
                                                        int shift, uint32_t *__restrict__ counts, uint32_t nblocks) {
    __shared__ uint32_t h[kRsWarps][256];
    for (int i = threadIdx.x; i < kRsWarps * 256; i += kRsThreads) (&h[0][0])[i] = 0;
    __syncthreads();
    const unsigned warp = threadIdx.x >> 5;
    const uint64_t base = (uint64_t)blockIdx.x * kRsThreads * kItems;
#pragma unroll 4
    for (int i = 0; i < kItems; ++i) {
        const uint64_t j = base + (uint64_t)i * kRsThreads + threadIdx.x;
        if (j < count) atomicAdd(&h[warp][(keys[j] >> shift) & 0xFF], 1u);
    }
    __syncthreads();
    for (int d = threadIdx.x; d < 256; d += kRsThreads) {
        uint32_t s = 0;
#pragma unroll
        for (int w = 0; w < kRsWarps; ++w) s += h[w][d];
        counts[(uint64_t)d * nblocks + blockIdx.x] = s;
    }
}

// Stable scatter: keys of a tile are taken round by round (round i holds
// entries base + i*256 + t), so input order is (round, thread).  A key's rank
// among equal digits = keys of that digit in earlier rounds + in earlier
// warps of this round + in earlier lanes of its warp.
template <int kItems>
__global__ void __launch_bounds__(kRsThreads) k_rs_scatter(const unsigned long long *__restrict__ in,
                                                           unsigned long long *__restrict__ out, uint64_t count,
                                                           int shift, const unsigned long long *__restrict__ offs,
                                                           uint32_t nblocks) {
    __shared__ uint32_t running[256];
    __shared__ uint32_t wc[kRsWarps][256];
    __shared__ unsigned long long start[256];
    const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
    for (int d = threadIdx.x; d < 256; d += kRsThreads) {
        running[d] = 0;
        start[d] = offs[(uint64_t)d * nblocks + blockIdx.x];
    }
    const uint64_t base = (uint64_t)blockIdx.x * kRsThreads * kItems;
    for (int i = 0; i < kItems; ++i) {
        for (int k = threadIdx.x; k < kRsWarps * 256; k += kRsThreads) (&wc[0][0])[k] = 0;
        __syncthreads();
        const uint64_t j = base + (uint64_t)i * kRsThreads + threadIdx.x;
        const bool valid = j < count;
        unsigned long long key = valid ? in[j] : 0ull;
        const uint32_t d = valid ? (uint32_t)((key >> shift) & 0xFF) : 256u + lane;  // invalid lanes: unique tags
        const unsigned peers = __match_any_sync(0xFFFFFFFFu, d);
        const uint32_t in_warp = __popc(peers & ((1u << lane) - 1u));
        if (valid && in_warp == 0) wc[warp][d] = __popc(peers);
        __syncthreads();
        if (valid) {
            uint32_t before = running[d] + in_warp;
            for (unsigned w = 0; w < warp; ++w) before += wc[w][d];
            out[start[d] + before] = key;
        }
        __syncthreads();
        for (int dd = threadIdx.x; dd < 256; dd += kRsThreads) {
            uint32_t s = 0;
#pragma unroll
            for (int w = 0; w < kRsWarps; ++w) s += wc[w][dd];
            running[dd] += s;
        }
        __syncthreads();
    }
}

__global__ void k_unique_flags(const unsigned long long *__restrict__ keys, uint64_t count, uint32_t *__restrict__ flag) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += stride)
        flag[i] = (i == 0 || keys[i] != keys[i - 1]) ? 1u : 0u;
}

__global__ void k_compact(const unsigned long long *__restrict__ keys, uint64_t count,
                          const uint32_t *__restrict__ flag, const unsigned long long *__restrict__ pos,
                          uint32_t *__restrict__ col, uint32_t *__restrict__ src32) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += stride) {
        if (!flag[i]) continue;
        const unsigned long long k = keys[i];
        col[pos[i]] = (uint32_t)k;
        src32[pos[i]] = (uint32_t)(k >> 32);
    }
}

// row_ptr[v] = first position p with src32[p] >= v (U = number of slots).
__global__ void k_rowptr(const uint32_t *__restrict__ src32, uint64_t U, uint32_t n, uint64_t *__restrict__ rp) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t p = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; p <= U; p += stride) {
        const uint64_t lo = p == 0 ? 0 : (uint64_t)src32[p - 1] + 1;   // first v whose start is p
        const uint64_t hi = p == U ? (uint64_t)n : (uint64_t)src32[p];  // last such v
        if (p == 0) {
            for (uint64_t v = 0; v <= hi && v <= n; ++v) rp[v] = 0;
        } else {
            for (uint64_t v = lo; v <= hi && v <= n; ++v) rp[v] = p;
        }
    }
}

__global__ void k_empty_rowptr(uint32_t n, uint64_t *__restrict__ rp) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t v = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; v <= n; v += stride) rp[v] = 0;
}

// ---------------------------------------------------------------------------- rows by counting

constexpr uint32_t kLaneRow = 32;      // entries of a row sorted by one lane
constexpr uint32_t kWarpRow = 1024;    // by its warp
constexpr uint32_t kBlockRow = 8192;   // by a block; longer rows go through bitmaps
constexpr uint32_t kMapN = 16384;      // up to this many vertices all rows that no warp sorts do
constexpr int kRowThreads = 256;
constexpr uint32_t kMapBits = 1u << 20;  // ids a bitmap covers (128 KB of shared memory)
// Rows whose bitmap lies in global memory: least entries, and how many (more of them keep every SM busy as it is).
// Two more launches, so only for many tuples (2^18 tuples of 2^22 vertices, one of them in every tuple: 0.48 against
// 0.43 ms, but every other build of that size 15 us less).
constexpr uint32_t kGiantRow = 1u << 17, kGiants = 64, kGiantTuples = 1u << 20;
constexpr uint32_t kNoPlace = 0xFFFFFFFFu;

// Entries before a vertex's newest one, one atomic per distinct vertex of the
// warp when neighbouring lanes meet on one (a hub named by most tuples).
__device__ __forceinline__ uint32_t take_place(uint32_t *cnt, uint32_t v, bool on) {
    const uint32_t w = on ? v : 0xFFFFFFFFu - lane_id();  // lanes without a vertex differ from all
    const bool met = __shfl_xor_sync(0xFFFFFFFFu, w, 1) == w;
    if (!__any_sync(0xFFFFFFFFu, met)) return on ? atomicAdd(&cnt[v], 1u) : 0u;
    const unsigned peers = __match_any_sync(0xFFFFFFFFu, w), leader = __ffs(peers) - 1;
    uint32_t at = 0;
    if (on && lane_id() == leader) at = atomicAdd(&cnt[v], (unsigned)__popc(peers));
    at = __shfl_sync(0xFFFFFFFFu, at, leader);
    return at + __popc(peers & ((1u << lane_id()) - 1u));
}

__global__ void k_count_entries(uint64_t t, const uint32_t *__restrict__ src, const uint32_t *__restrict__ dst,
                                uint32_t n, uint32_t *__restrict__ cnt, uint32_t *__restrict__ place_a,
                                uint32_t *__restrict__ place_b, Ctl *ctl) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    const uint64_t t_round = (t + 31) & ~uint64_t(31);
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < t_round; i += stride) {
        uint32_t a = 0, b = 0;
        bool keep = false;
        if (i < t) {
            a = src[i];
            b = dst[i];
            if (a >= n || b >= n) ctl->error = 1;
            else keep = a != b;
        }
        const uint32_t pa = take_place(cnt, a, keep), pb = take_place(cnt, b, keep);
        if (i < t) {
            place_a[i] = keep ? pa : kNoPlace;
            place_b[i] = keep ? pb : kNoPlace;
        }
    }
}

// Few vertices named by many tuples: the atomics of k_count_entries meet on few
// addresses, so a block counts kFewTile tuples in shared memory and takes its places
// of a vertex from the counts at once.  2^24 tuples of 8 / 256 / 1024 vertices, whole builds:
// 5.5 / 7.9 / 3.0 -> 0.68 / 0.63 / 0.61 ms (the radix sort 1.3 / 1.8 / 2.4); at fewer than 16 tuples
// a vertex or 2^16 in all it is no faster.
constexpr uint32_t kFewN = 8192, kFewTile = 8192, kFewFrom = 1u << 16;
__global__ void __launch_bounds__(1024) k_count_few(uint64_t t, const uint32_t *__restrict__ src,
                                                    const uint32_t *__restrict__ dst, uint32_t n,
                                                    uint32_t *__restrict__ cnt, uint32_t *__restrict__ place_a,
                                                    uint32_t *__restrict__ place_b, Ctl *ctl) {
    __shared__ uint32_t local[kFewN];  // entries of the tile per vertex, then the first one's place
    constexpr int kItems = kFewTile / 1024;
    for (uint64_t lo = (uint64_t)blockIdx.x * kFewTile; lo < t; lo += (uint64_t)gridDim.x * kFewTile) {
        for (uint32_t v = threadIdx.x; v < n; v += 1024) local[v] = 0;
        __syncthreads();
        uint32_t a[kItems], b[kItems], pa[kItems], pb[kItems];
#pragma unroll
        for (int k = 0; k < kItems; ++k) {
            const uint64_t i = lo + 1024 * k + threadIdx.x;
            a[k] = i < t ? src[i] : 0u;
            b[k] = i < t ? dst[i] : 0u;
        }
#pragma unroll
        for (int k = 0; k < kItems; ++k) {
            if (a[k] >= n || b[k] >= n) {
                ctl->error = 1;
                a[k] = b[k] = 0;
            }
            pa[k] = take_place(local, a[k], a[k] != b[k]);
            pb[k] = take_place(local, b[k], a[k] != b[k]);
        }
        __syncthreads();
        for (uint32_t v = threadIdx.x; v < n; v += 1024) {
            const uint32_t c = local[v];
            if (c) local[v] = atomicAdd(&cnt[v], c);
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kItems; ++k) {
            const uint64_t i = lo + 1024 * k + threadIdx.x;
            if (i < t) {
                place_a[i] = a[k] != b[k] ? local[a[k]] + pa[k] : kNoPlace;
                place_b[i] = a[k] != b[k] ? local[b[k]] + pb[k] : kNoPlace;
            }
        }
        __syncthreads();
    }
}

__global__ void k_place_entries(uint64_t t, const uint32_t *__restrict__ src, const uint32_t *__restrict__ dst,
                                const uint64_t *__restrict__ start, const uint32_t *__restrict__ place_a,
                                const uint32_t *__restrict__ place_b, uint32_t *__restrict__ raw) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < t; i += stride) {
        const uint32_t pa = place_a[i], pb = place_b[i];
        if (pa == kNoPlace) continue;
        const uint32_t a = src[i], b = dst[i];
        raw[start[a] + pa] = b;
        raw[start[b] + pb] = a;
    }
}

// Rows of up to kWarpRow entries: sorted in place, repeats dropped; deg[v] =
// entries left.  Longer rows are listed for a block each, or for the bitmaps.
// Lanes own rows of up to kLaneRow entries (insertion sort in their column of
// the warp's buffer), the warp takes the others one by one.
__global__ void __launch_bounds__(kRowThreads) k_sort_rows(uint32_t n, const uint64_t *__restrict__ start,
                                                           uint32_t *__restrict__ raw, uint32_t *__restrict__ deg,
                                                           uint32_t *__restrict__ big, uint32_t *__restrict__ huge,
                                                           uint32_t per_warp, uint32_t grab, uint32_t block_row, Ctl *ctl) {
    __shared__ __align__(16) uint32_t sbuf[kRowThreads / 32][kWarpRow];
    const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    uint32_t *buf = sbuf[warp];
    uint32_t top = 0;
    const uint64_t chunks = ((uint64_t)n + per_warp - 1) / per_warp;
    uint32_t c = 0, left = 0;
    for (;; ++c) {
        if (left == 0) {  // the next `grab` chunks (one by one, the atomics of 2^21 chunks take 1.6 ms)
            if (lane == 0) c = atomicAdd(&ctl->fill_next, grab);
            c = __shfl_sync(0xFFFFFFFFu, c, 0);
            left = grab;
        }
        --left;
        if (c >= chunks) break;
        const uint64_t x = (uint64_t)c * per_warp + lane;
        const bool valid = lane < per_warp && x < n;
        const uint64_t b = valid ? start[x] : 0;
        const uint64_t d64 = valid ? start[x + 1] - b : 0;
        const uint32_t d = (uint32_t)d64;
        if (valid && d <= kLaneRow) {
            uint32_t k = 0;
            for (uint32_t j0 = 0; j0 < d; j0 += 8) {
                uint32_t y[8];
#pragma unroll
                for (uint32_t t = 0; t < 8; ++t) y[t] = j0 + t < d ? raw[b + j0 + t] : 0u;
#pragma unroll
                for (uint32_t t = 0; t < 8; ++t) {
                    if (j0 + t >= d) break;
                    uint32_t i = k;
                    while (i > 0 && buf[(i - 1) * 32 + lane] > y[t]) --i;
                    if (i > 0 && buf[(i - 1) * 32 + lane] == y[t]) continue;  // a repeat
                    for (uint32_t m = k; m > i; --m) buf[m * 32 + lane] = buf[(m - 1) * 32 + lane];
                    buf[i * 32 + lane] = y[t];
                    ++k;
                }
            }
            for (uint32_t i = 0; i < k; ++i) raw[b + i] = buf[i * 32 + lane];
            deg[x] = k;
            top = k > top ? k : top;
        }
        __syncwarp();
        if (valid && d > kWarpRow) {
            if (d <= block_row) big[atomicAdd(&ctl->n_big, 1u)] = (uint32_t)x;
            else huge[atomicAdd(&ctl->n_huge, 1u)] = (uint32_t)x;
        }
        unsigned pending = __ballot_sync(0xFFFFFFFFu, valid && d > kLaneRow && d <= kWarpRow);
        while (pending) {
            const int src = __ffs(pending) - 1;
            pending &= pending - 1;
            const uint32_t bd = __shfl_sync(0xFFFFFFFFu, d, src);
            const uint64_t bb = __shfl_sync(0xFFFFFFFFu, b, src);
            for (uint32_t j = lane; j < bd; j += 32) buf[j] = raw[bb + j];
            __syncwarp();
            warp_sort_any(buf, bd);
            uint32_t k = 0;
            for (uint32_t j0 = 0; j0 < bd; j0 += 32) {
                const uint32_t j = j0 + lane;
                const bool keep = j < bd && (j == 0 || buf[j] != buf[j - 1]);
                const unsigned m = __ballot_sync(0xFFFFFFFFu, keep);
                if (keep) raw[bb + k + __popc(m & lt)] = buf[j];
                k += __popc(m);
            }
            if (lane == 0) deg[(uint64_t)c * per_warp + src] = k;
            top = k > top ? k : top;
            __syncwarp();
        }
    }
    top = __reduce_max_sync(0xFFFFFFFFu, top);
    if (lane == 0 && top) atomicMax(&ctl->max_s2, top);
}

// Exclusive position of this thread's flag among the block's (all threads; two barriers).
__device__ __forceinline__ uint32_t block_rank(bool flag, uint32_t *warp_cnt, uint32_t *total) {
    const unsigned lane = lane_id(), warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const unsigned m = __ballot_sync(0xFFFFFFFFu, flag);
    if (lane == 0) warp_cnt[warp] = __popc(m);
    __syncthreads();
    uint32_t v = lane < nw ? warp_cnt[lane] : 0u, incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= (unsigned)o) incl += y;
    }
    const uint32_t before = __shfl_sync(0xFFFFFFFFu, incl - v, warp);
    *total = __shfl_sync(0xFFFFFFFFu, incl, 31);
    __syncthreads();
    return before + __popc(m & ((1u << lane) - 1u));
}

// Rows of kWarpRow + 1 .. kBlockRow entries: a block each sorts the row in
// shared memory and writes its distinct entries back.  Its warps sort runs of
// 1024 in registers; a merge starts with a mirrored compare over the block (both
// runs ascending), and its steps below 1024 are the warps' own again, so a row of
// 8192 meets 12 barriers instead of the 91 of a plain bitonic network (R-MAT 21:
// 1.00 -> 0.42 ms for all these rows).
__device__ __forceinline__ void compare_swap(uint32_t *sb, uint32_t i, uint32_t l) {
    const uint32_t u = sb[i], w = sb[l];
    if (u > w) {
        sb[i] = w;
        sb[l] = u;
    }
}

__global__ void __launch_bounds__(256) k_sort_rows_big(const uint64_t *__restrict__ start, uint32_t *__restrict__ raw,
                                                       uint32_t *__restrict__ deg, const uint32_t *__restrict__ big,
                                                       Ctl *ctl) {
    __shared__ __align__(16) uint32_t sb[kBlockRow];
    __shared__ uint32_t warp_cnt[32];
    __shared__ unsigned int s_i;
    const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
    uint32_t *run = sb + 1024 * warp;  // eight warps, 1024 keys each
    const uint32_t nb = ctl->n_big;
    for (;;) {
        if (threadIdx.x == 0) s_i = atomicAdd(&ctl->sort_next, 1u);
        __syncthreads();
        const uint32_t i = s_i;
        if (i >= nb) break;
        const uint32_t x = big[i];
        const uint64_t b = start[x];
        const uint32_t d = (uint32_t)(start[x + 1] - b);
        uint32_t P = 2048;
        while (P < d) P <<= 1;
        const bool mine = 1024 * warp < P;
        const uint32_t left = d > 1024 * warp ? d - 1024 * warp : 0u;
        if (mine) {
            for (uint32_t t = lane; t < 1024; t += 32) run[t] = t < left ? raw[b + 1024 * warp + t] : kEmpty;
            __syncwarp();
            warp_sort_large(run, left < 1024 ? left : 1024u, 1024u);
        }
        for (uint32_t k = 2048; k <= P; k <<= 1) {
            __syncthreads();
            for (uint32_t p = threadIdx.x; p < P / 2; p += blockDim.x) {  // mirrored halves of every k keys
                const uint32_t base = (p / (k / 2)) * k, o = p & (k / 2 - 1);
                compare_swap(sb, base + o, base + k - 1 - o);
            }
            for (uint32_t j = k / 4; j >= 1024; j >>= 1) {
                __syncthreads();
                for (uint32_t p = threadIdx.x; p < P / 2; p += blockDim.x) {
                    const uint32_t e = ((p & ~(j - 1)) << 1) | (p & (j - 1));
                    compare_swap(sb, e, e | j);
                }
            }
            __syncthreads();
            if (mine) {
                for (uint32_t j = 512; j >= 256; j >>= 1) {
                    for (uint32_t p = lane; p < 512; p += 32) {
                        const uint32_t e = ((p & ~(j - 1)) << 1) | (p & (j - 1));
                        compare_swap(run, e, e | j);
                    }
                    __syncwarp();
                }
                for (uint32_t c = 0; c < 1024; c += 256) warp_merge_256(run + c, false);
            }
        }
        __syncthreads();
        uint32_t kept = 0;
        for (uint32_t j0 = 0; j0 < d; j0 += blockDim.x) {
            const uint32_t j = j0 + threadIdx.x;
            const bool keep = j < d && (j == 0 || sb[j] != sb[j - 1]);
            uint32_t total;
            const uint32_t at = block_rank(keep, warp_cnt, &total);
            if (keep) raw[b + kept + at] = sb[j];
            kept += total;
        }
        if (threadIdx.x == 0) {
            deg[x] = kept;
            atomicMax(&ctl->max_s2, kept);
        }
        __syncthreads();
    }
}

// The first kGiants rows of `giant` entries or more among the listed ones, and their
// bitmaps cleared.  Every block finds them, the first one writes them down: every listed
// row learns the number of its bitmap (kNoPlace: none) behind the list of big rows (a
// row is in one of the two lists, so they do not meet).  Apart from k_sort_rows, which the
// few lines slow down by a tenth.
__global__ void __launch_bounds__(1024) k_list_giants(uint32_t n, const uint64_t *__restrict__ start,
                                                      const uint32_t *__restrict__ huge, uint32_t *__restrict__ big,
                                                      uint32_t *__restrict__ giants, uint32_t giant,
                                                      uint32_t *__restrict__ maps, uint32_t giant_words, Ctl *ctl) {
    __shared__ uint32_t warp_cnt[32];
    const uint32_t nh = ctl->n_huge;
    uint32_t ng = 0;
    for (uint32_t i0 = 0; i0 < nh; i0 += 1024) {
        const uint32_t i = i0 + threadIdx.x, x = i < nh ? huge[i] : 0u;
        const bool is = i < nh && start[x + 1] - start[x] >= giant;
        uint32_t total;
        const uint32_t g = ng + block_rank(is, warp_cnt, &total);
        if (blockIdx.x == 0) {
            if (is && g < kGiants) giants[g] = x;
            if (i < nh) big[n - 1 - i] = is && g < kGiants ? g : kNoPlace;
        }
        ng += total;
    }
    ng = min(ng, kGiants);
    if (blockIdx.x == 0 && threadIdx.x == 0) ctl->n_giant = ng;
    for (uint64_t i = (uint64_t)blockIdx.x * 1024 + threadIdx.x; i < (uint64_t)ng * giant_words; i += 1024ull * gridDim.x)
        maps[i] = 0;
}

// The ids of the giant rows, marked in bitmaps in global memory (L2) by the whole grid: a
// block of k_map_rows reads 2.3 entries a clock, so a vertex named by most tuples kept a
// few blocks busy and the others idle (2^24 tuples of 2^22 vertices, one of them in every
// tuple: 17.4 -> 1.9 ms; the radix sort 3.1).  A warp takes 1024 entries; set bits are not set again.
__global__ void __launch_bounds__(256) k_mark_giant(const uint64_t *__restrict__ start,
                                                    const uint32_t *__restrict__ raw,
                                                    const uint32_t *__restrict__ giants, uint32_t *maps,
                                                    uint32_t giant_words, const Ctl *ctl) {
    const uint32_t ng = ctl->n_giant;
    const uint64_t warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    const uint64_t w0 = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    for (uint32_t g = 0; g < ng; ++g) {
        uint32_t *map = maps + (uint64_t)g * giant_words;
        const uint64_t b = start[giants[g]], e = start[giants[g] + 1];
        for (uint64_t j0 = b + 1024 * w0; j0 < e; j0 += 1024 * warps) {
#pragma unroll
            for (uint32_t k = 0; k < 1024; k += 256) {
                uint32_t y[8], m[8];
#pragma unroll
                for (uint32_t t = 0; t < 8; ++t) {
                    const uint64_t j = j0 + k + 32 * t + lane_id();
                    y[t] = raw[j < e ? j : b];
                }
#pragma unroll
                for (uint32_t t = 0; t < 8; ++t) m[t] = __ldcg(map + (y[t] >> 5));
#pragma unroll
                for (uint32_t t = 0; t < 8; ++t)
                    if (!((m[t] >> (y[t] & 31u)) & 1u)) atomicOr(map + (y[t] >> 5), 1u << (y[t] & 31u));
            }
        }
    }
}

// Longer rows: one block per (row, range of kMapBits ids) marks the row's ids of
// its range in a bitmap (a giant row's are marked already).  kEmit = false counts them (parts, deg); kEmit = true,
// once the rows' places are known, writes them out in order.
template <bool kEmit>
__global__ void __launch_bounds__(1024) k_map_rows(uint32_t n, const uint64_t *__restrict__ start,
                                                   const uint32_t *__restrict__ raw, const uint32_t *__restrict__ huge,
                                                   const uint32_t *__restrict__ big, const uint32_t *__restrict__ maps,
                                                   uint32_t giant_words, uint32_t ranges, uint32_t *__restrict__ parts,
                                                   uint32_t *__restrict__ deg, const uint64_t *__restrict__ rp,
                                                   uint32_t *__restrict__ col, Ctl *ctl) {
    extern __shared__ uint32_t map[];  // kMapBits bits
    __shared__ uint32_t warp_cnt[32];
    const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
    const uint64_t units = (uint64_t)ctl->n_huge * ranges;
    for (uint64_t unit = blockIdx.x; unit < units; unit += gridDim.x) {
        const uint32_t x = huge[unit / ranges], range = (uint32_t)(unit % ranges), lo = range * kMapBits;
        const uint64_t b = start[x], e = start[x + 1];
        const uint32_t words = (min(n - lo, kMapBits) + 31) / 32;
        const uint32_t giant = maps ? big[n - 1 - (uint32_t)(unit / ranges)] : kNoPlace;
        if (giant != kNoPlace) {
            const uint32_t *m = maps + (uint64_t)giant * giant_words + lo / 32;
            for (uint32_t i = threadIdx.x; i < words; i += blockDim.x) map[i] = m[i];
        } else {
            for (uint32_t i = threadIdx.x; i < words; i += blockDim.x) map[i] = 0;
            __syncthreads();
            for (uint64_t j0 = b + threadIdx.x; j0 < e; j0 += 16 * blockDim.x) {  // sixteen in flight (one: half the rate)
                uint32_t y[16];
#pragma unroll
                for (uint32_t t = 0; t < 16; ++t) {
                    const uint64_t j = j0 + t * blockDim.x;
                    y[t] = j < e ? raw[j] - lo : kMapBits;
                }
#pragma unroll
                for (uint32_t t = 0; t < 16; ++t)
                    if (y[t] < kMapBits && !((map[y[t] >> 5] >> (y[t] & 31u)) & 1u))
                        atomicOr(&map[y[t] >> 5], 1u << (y[t] & 31u));
            }
        }
        __syncthreads();
        // every thread owns a run of words: its ids come after those of the threads before
        const uint32_t per = (words + blockDim.x - 1) / blockDim.x, w0 = threadIdx.x * per;
        uint32_t mine = 0;
        for (uint32_t i = w0; i < min(w0 + per, words); ++i) mine += __popc(map[i]);
        uint32_t incl = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
            if (lane >= (unsigned)o) incl += y;
        }
        if (lane == 31) warp_cnt[warp] = incl;
        __syncthreads();
        uint32_t v = warp_cnt[lane], wi = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, wi, o);
            if (lane >= (unsigned)o) wi += y;
        }
        const uint32_t before = __shfl_sync(0xFFFFFFFFu, wi - v, warp), total = __shfl_sync(0xFFFFFFFFu, wi, 31);
        if constexpr (kEmit) {
            uint64_t at = rp[x] + before + incl - mine;
            for (uint32_t r = 0; r < range; ++r) at += parts[unit - range + r];
            for (uint32_t i = w0; i < min(w0 + per, words); ++i)
                for (uint32_t m = map[i]; m; m &= m - 1) col[at++] = lo + 32 * i + __ffs(m) - 1;
        } else if (threadIdx.x == 0) {
            parts[unit] = total;
            atomicMax(&ctl->max_s2, atomicAdd(&deg[x], total) + total);
        }
        __syncthreads();
    }
}

// The sorted rows (bitmap rows aside) into their final places: a warp flattens
// the entries of 32 rows, one per lane and step (their places are contiguous).
__global__ void __launch_bounds__(256) k_pack_rows(uint32_t n, const uint64_t *__restrict__ start,
                                                   const uint32_t *__restrict__ raw, const uint64_t *__restrict__ rp,
                                                   uint32_t *__restrict__ col, uint32_t block_row) {
    const unsigned lane = lane_id();
    const uint64_t warps = ((uint64_t)gridDim.x * blockDim.x) >> 5, groups = ((uint64_t)n + 31) / 32;
    for (uint64_t g = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; g < groups; g += warps) {
        const uint64_t x = g * 32 + lane;
        uint64_t b = 0, to = 0;
        uint32_t d = 0;
        if (x < n) {
            b = start[x];
            to = rp[x];
            d = (uint32_t)(rp[x + 1] - to);
            if (start[x + 1] - b > block_row) d = 0;
        }
        uint32_t incl = d;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
            if (lane >= (unsigned)o) incl += y;
        }
        const uint32_t total = __shfl_sync(0xFFFFFFFFu, incl, 31);
        const uint64_t from0 = b - (incl - d), to0 = to - (incl - d);  // minus the row's first flat position
        for (uint32_t e0 = 0; e0 < total; e0 += 32) {
            const uint32_t e = e0 + lane;
            uint32_t r = 0;  // the row of flat position e: the first whose inclusive count passes it
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                if (__shfl_sync(0xFFFFFFFFu, incl, r + o - 1) <= e) r += o;
            const uint64_t f = __shfl_sync(0xFFFFFFFFu, from0, r), w = __shfl_sync(0xFFFFFFFFu, to0, r);
            if (e < total) col[w + e] = raw[f + e];
        }
    }
}

// Well-formedness: monotone row_ptr ending at `slots`, ids < n, rows strictly
// ascending (no repeats), no self-loops, and every (v, w) has its (w, v).
__global__ void k_validate(uint32_t n, const uint64_t *__restrict__ rp, const uint32_t *__restrict__ col,
                           uint64_t slots, Ctl *ctl) {
    const unsigned lane = lane_id();
    const uint64_t warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    for (uint64_t v = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; v < n; v += warps) {
        const uint64_t b = rp[v], e = rp[v + 1];
        if (e < b || e > slots || (v == 0 && b != 0) || (v + 1 == n && e != slots)) {
            if (lane == 0) ctl->error = 1;
            continue;
        }
        for (uint64_t j = b + lane; j < e; j += 32) {
            const uint32_t w = col[j];
            bool bad = w >= n || w == v || (j > b && col[j - 1] >= w);
            if (!bad) {
                uint64_t lo = rp[w], hi = rp[w + 1];
                if (hi > slots || lo > hi) {  // w's own row is malformed: never read outside col
                    ctl->error = 1;
                    continue;
                }
                bool found = false;
                while (lo < hi) {
                    const uint64_t mid = (lo + hi) >> 1;
                    const uint32_t x = col[mid];
                    if (x == v) { found = true; break; }
                    if (x < v) lo = mid + 1; else hi = mid;
                }
                bad = !found;
            }
            if (bad) ctl->error = 1;
        }
    }
}

__global__ void k_max_deg(uint32_t n, const uint64_t *__restrict__ rp, Ctl *ctl) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    unsigned m = 0;
    for (uint64_t v = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
        const uint64_t d = rp[v + 1] - rp[v];
        const unsigned dd = d > 0xFFFFFFFFull ? 0xFFFFFFFFu : (unsigned)d;
        m = dd > m ? dd : m;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        unsigned y = __shfl_xor_sync(0xFFFFFFFFu, m, o);
        m = y > m ? y : m;
    }
    if (lane_id() == 0 && m) atomicMax(&ctl->max_s2, m);
}

__global__ void k_ctl_zero(Ctl *ctl) {
    unsigned int *w = reinterpret_cast<unsigned int *>(ctl);
    for (unsigned i = threadIdx.x; i < sizeof(Ctl) / 4; i += blockDim.x) w[i] = 0;
}

unsigned grid_for(uint64_t work, unsigned threads, unsigned cap) {
    uint64_t b = (work + threads - 1) / threads;
    if (b < 1) b = 1;
    if (b > cap) b = cap;
    return (unsigned)b;
}

tc_status pull(tc_ctx *ctx) {
    TC_CUDA(ctx, cudaMemcpyAsync(ctx->h_ctl, ctx->d_ctl, sizeof(Ctl), cudaMemcpyDeviceToHost, ctx->stream));
    TC_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    return TC_OK;
}

}  // namespace

uint64_t radix_tiles(uint64_t count) { return (count + rs_tile(count) - 1) / rs_tile(count); }
uint64_t radix_tiles_cap(uint64_t count) {
    return std::max(radix_tiles(count), radix_tiles(std::min<uint64_t>(count, kRsShort)));
}

uint32_t radix_sort_u64(unsigned long long **cur, unsigned long long **alt, uint64_t count, const int *shifts,
                        int nshifts, uint32_t *counts, uint64_t *coffs, uint64_t *tmp, cudaStream_t s) {
    if (count < 2) return 0;
    const uint32_t nblk = (uint32_t)radix_tiles(count);
    uint32_t launches = 0;
    const bool few = count <= kRsShort;
    auto k_rs_hist = few ? tc::k_rs_hist<kRsItemsShort> : tc::k_rs_hist<kRsItems>;
    auto k_rs_scatter = few ? tc::k_rs_scatter<kRsItemsShort> : tc::k_rs_scatter<kRsItems>;
    for (int i = 0; i < nshifts; ++i) {
        k_rs_hist<<<nblk, kRsThreads, 0, s>>>(*cur, count, shifts[i], counts, nblk);
        launches += 2 + scan_u32_to_u64(counts, coffs, 256ull * nblk, tmp, s);
        k_rs_scatter<<<nblk, kRsThreads, 0, s>>>(*cur, *alt, count, shifts[i],
                                                 reinterpret_cast<const unsigned long long *>(coffs), nblk);
        std::swap(*cur, *alt);
    }
    return launches;
}

// Tuples and vertices the counting build takes: 32-bit places, at most 64 bitmap ranges.
constexpr uint64_t kCountTuples = 1ull << 31;
constexpr uint32_t kCountN = 1u << 26;

// Few tuples over very many vertices: the counting build passes over the vertices eight
// times, the sort once.  Radix sort / counting: 2^24 vertices, 2^17 / 2^20 / 2^21 tuples 0.51 / 0.58 /
// 0.74 against 0.59 / 0.66 / 0.72 ms, 2^26 and 2^14 / 2^20 / 2^22 / 2^24 1.0 / 1.1 / 1.8 / 4.8 against 1.5 / 1.8 /
// 2.2 / 4.6 (2^22 vertices 0.42 against 0.30 at 2^16 tuples); with 2^10 tuples its row_ptr has runs
// that one thread each fills: 5.9 against 1.5.
static bool sparse_tuples(uint32_t n, uint64_t t) { return n >= (1u << 24) && t <= n / 16 && t > n / 8192; }

static tc_status build_csr_counting(tc_ctx *ctx, uint32_t n, uint64_t t, const uint32_t *d_src, const uint32_t *d_dst,
                                    uint64_t **rp_out, uint32_t **col_out, uint64_t *slots_out, bool *pooled_out,
                                    uint32_t *max_deg, bool *no_room) {
    cudaStream_t s = ctx->stream;
    const unsigned cap = (unsigned)ctx->num_sms * 16u;
    const uint32_t ranges = (n + kMapBits - 1) / kMapBits;
    // the longest row a block sorts: of few vertices a bitmap is shorter (2^20 tuples of 1024 vertices 0.41 -> 0.17 ms)
    const uint32_t block_row = n <= kMapN ? kWarpRow : kBlockRow;
    const uint64_t max_huge = 2 * t / block_row + 1;  // rows of more entries
    // rows of at least n / 16 entries: at most 32 t / n bitmaps of n / 8 bytes, which the places' 8 t bytes hold
    // once the entries are placed
    const uint32_t giant = std::max(kGiantRow, n / 16), giant_words = (n + 31) / 32;
    const bool giants = t >= kGiantTuples && 2 * t >= giant;
    auto r = [](size_t b) { return (b + 255) & ~size_t(255); };
    const size_t n1 = (size_t)n + 1;
    const size_t need = 4 * r(4 * n1) + r(8 * n1) + 2 * r(8 * t) + r(4 * max_huge * ranges) +
                        r(8 * scan_tmp_elems(n1)) + 4096;
    tc_status st = arena_reserve(ctx, need);
    *no_room = st == TC_ERR_OOM;
    if (st != TC_OK) return st;
    Arena &a = ctx->arena;
    a.reset();
    auto *cnt = a.take<uint32_t>(n1);
    auto *deg = a.take<uint32_t>(n1);
    auto *big = a.take<uint32_t>(n1);
    auto *huge = a.take<uint32_t>(n1);
    auto *start = a.take<uint64_t>(n1);
    auto *place_a = a.take<uint32_t>(2 * t);
    uint32_t *place_b = place_a + t, *maps = giants ? place_a : nullptr;
    auto *raw = a.take<uint32_t>(2 * t);
    auto *parts = a.take<uint32_t>(max_huge * ranges);
    auto *tmp = a.take<uint64_t>(scan_tmp_elems(n1));
    if (!cnt || !deg || !big || !huge || !start || !place_a || !raw || !parts || !tmp)
        return set_error(ctx, TC_ERR_OOM, "arena carve failed (build_csr)");
    uint64_t *rp = nullptr;
    uint32_t *col = nullptr;
    bool pooled = false, pooled2 = false;
    if (graph_alloc(ctx, (void **)&rp, sizeof(uint64_t) * n1, &pooled) != cudaSuccess) {
        cudaGetLastError();
        return set_error(ctx, TC_ERR_OOM, "tc_build_csr: row_ptr allocation failed");
    }
    *pooled_out = pooled;
    k_ctl_zero<<<1, 128, 0, s>>>(ctx->d_ctl);
    cudaError_t e = cudaMemsetAsync(cnt, 0, 4 * n1, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(deg, 0, 4 * n1, s);
    if (n <= kFewN && t >= kFewFrom && t >= 16ull * n)
        k_count_few<<<grid_for(t, kFewTile, cap), 1024, 0, s>>>(t, d_src, d_dst, n, cnt, place_a, place_b, ctx->d_ctl);
    else
        k_count_entries<<<grid_for(t, 256, cap), 256, 0, s>>>(t, d_src, d_dst, n, cnt, place_a, place_b, ctx->d_ctl);
    scan_u32_to_u64(cnt, start, n, tmp, s);
    k_place_entries<<<grid_for(t, 256, cap), 256, 0, s>>>(t, d_src, d_dst, start, place_a, place_b, raw);
    // long rows of small graphs spread out (2^18 tuples of 512 vertices 0.32 -> 0.22 ms by one vertex a warp)
    const uint32_t per_warp = n >= (1u << 20) ? 32u : n >= (1u << 18) ? 16u : n > kFewN ? 8u : n > 1024 ? 2u : 1u;
    // an eighth of a warp's share of the chunks
    const uint32_t grab = std::max(1u, std::min(16u, n / (32u * 8u * (kRowThreads / 32) * cap)));
    k_sort_rows<<<grid_for((uint64_t)n * (32 / per_warp), kRowThreads, cap), kRowThreads, 0, s>>>(
        n, start, raw, deg, big, huge, per_warp, grab, block_row, ctx->d_ctl);
    const bool bigs = 2 * t > kWarpRow, huges = 2 * t > block_row;  // there may be some
    const int map_smem = (int)(kMapBits / 8);
    if (bigs) k_sort_rows_big<<<(unsigned)ctx->num_sms * 6u, 256, 0, s>>>(start, raw, deg, big, ctx->d_ctl);
    if (giants) {
        k_list_giants<<<(unsigned)ctx->num_sms, 1024, 0, s>>>(n, start, huge, big, cnt, giant, maps, giant_words,
                                                              ctx->d_ctl);
        k_mark_giant<<<(unsigned)ctx->num_sms * 8u, 256, 0, s>>>(start, raw, cnt, maps, giant_words, ctx->d_ctl);
    }
    if (huges) {
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k_map_rows<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, map_smem);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k_map_rows<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, map_smem);
        k_map_rows<false><<<(unsigned)ctx->num_sms, 1024, map_smem, s>>>(
            n, start, raw, huge, big, maps, giant_words, ranges, parts, deg, nullptr, nullptr, ctx->d_ctl);
    }
    scan_u32_to_u64(deg, rp, n, tmp, s);
    uint64_t U = 0;
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(&U, rp + n, sizeof(uint64_t), cudaMemcpyDeviceToHost, s);
    if (e != cudaSuccess) {
        graph_free(ctx, rp, pooled);
        return cuda_error(ctx, e, "tc_build_csr kernels");
    }
    st = pull(ctx);
    if (st == TC_OK && ctx->h_ctl->error) st = set_error(ctx, TC_ERR_INVALID, "tc_build_csr: a tuple names a vertex id >= n");
    if (st != TC_OK) {
        graph_free(ctx, rp, pooled);
        return st;
    }
    *max_deg = ctx->h_ctl->max_s2;
    if (graph_alloc(ctx, (void **)&col, sizeof(uint32_t) * (size_t)(U + 1), &pooled2) != cudaSuccess) {
        cudaGetLastError();
        graph_free(ctx, rp, pooled);
        return set_error(ctx, TC_ERR_OOM, "tc_build_csr: col allocation failed");
    }
    if (U) {
        k_pack_rows<<<grid_for(n, 256, cap), 256, 0, s>>>(n, start, raw, rp, col, block_row);
        if (ctx->h_ctl->n_huge)
            k_map_rows<true><<<(unsigned)ctx->num_sms, 1024, map_smem, s>>>(
                n, start, raw, huge, big, maps, giant_words, ranges, parts, deg, rp, col, ctx->d_ctl);
    }
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) {
        graph_free(ctx, rp, pooled);
        graph_free(ctx, col, pooled2);
        return cuda_error(ctx, e, "tc_build_csr kernels");
    }
    *rp_out = rp;
    *col_out = col;
    *slots_out = U;
    return TC_OK;
}

tc_status build_csr_device(tc_ctx *ctx, uint32_t n, uint64_t t, const uint32_t *d_src, const uint32_t *d_dst,
                           uint64_t **rp_out, uint32_t **col_out, uint64_t *slots_out, bool *pooled_out,
                           uint32_t *max_deg) {
    if (t && t < kCountTuples && n && n <= kCountN && !sparse_tuples(n, t)) {
        bool no_room = false;
        const tc_status st =
            build_csr_counting(ctx, n, t, d_src, d_dst, rp_out, col_out, slots_out, pooled_out, max_deg, &no_room);
        if (!no_room) return st;  // (its scratch grows with the vertices, the sort's does not)
    }
    cudaStream_t s = ctx->stream;
    const unsigned cap = (unsigned)ctx->num_sms * 16u;
    const uint64_t K = 2 * t;  // upper bound on keys
    const uint64_t nblk_max = radix_tiles_cap(K);
    auto r = [](size_t b) { return (b + 255) & ~size_t(255); };
    const size_t need = 2 * r(8 * (K + 1)) + r(4 * (K + 1)) + r(8 * (K + 2)) + r(4 * (K + 1)) +
                        r(4 * (256 * nblk_max + 1)) + r(8 * (256 * nblk_max + 2)) +
                        r(8 * scan_tmp_elems(std::max<uint64_t>(K, 256 * nblk_max) + 2)) + 4096;
    tc_status st = arena_reserve(ctx, need);
    if (st != TC_OK) return st;
    Arena &a = ctx->arena;
    a.reset();
    auto *k0 = a.take<unsigned long long>(K + 1);
    auto *k1 = a.take<unsigned long long>(K + 1);
    auto *flag = a.take<uint32_t>(K + 1);
    auto *pos = a.take<uint64_t>(K + 2);
    auto *src32 = a.take<uint32_t>(K + 1);
    auto *counts = a.take<uint32_t>(256 * nblk_max + 1);
    auto *coffs = a.take<uint64_t>(256 * nblk_max + 2);
    auto *tmp = a.take<uint64_t>(scan_tmp_elems(std::max<uint64_t>(K, 256 * nblk_max) + 2));
    if (!k0 || !k1 || !flag || !pos || !src32 || !counts || !coffs || !tmp)
        return set_error(ctx, TC_ERR_OOM, "arena carve failed (build_csr)");

    k_ctl_zero<<<1, 128, 0, s>>>(ctx->d_ctl);
    if (t) k_make_keys<<<grid_for(t, 256, cap), 256, 0, s>>>(t, d_src, d_dst, n, k0, ctx->d_ctl);
    TC_CUDA(ctx, cudaGetLastError());
    st = pull(ctx);
    if (st != TC_OK) return st;
    if (ctx->h_ctl->error) return set_error(ctx, TC_ERR_INVALID, "tc_build_csr: a tuple names a vertex id >= n");
    const uint64_t nk = ctx->h_ctl->visited_edges;  // keys written (2 per kept tuple)

    // significant bits of an id: the radix passes cover [0, B) and [32, 32 + B)
    int B = 0;
    while (B < 32 && (1ull << B) < n) ++B;
    std::vector<int> shifts;
    for (int sh = 0; sh < B; sh += 8) shifts.push_back(sh);
    for (int sh = 0; sh < B; sh += 8) shifts.push_back(32 + sh);
    unsigned long long *cur = k0, *alt = k1;
    radix_sort_u64(&cur, &alt, nk, shifts.data(), (int)shifts.size(), counts, coffs, tmp, s);
    uint64_t *rp = nullptr;
    uint32_t *col = nullptr;
    uint64_t U = 0;
    if (nk) {
        k_unique_flags<<<grid_for(nk, 256, cap), 256, 0, s>>>(cur, nk, flag);
        scan_u32_to_u64(flag, pos, nk, tmp, s);
        TC_CUDA(ctx, cudaMemcpyAsync(&U, pos + nk, sizeof(uint64_t), cudaMemcpyDeviceToHost, s));
        TC_CUDA(ctx, cudaStreamSynchronize(s));
    }
    bool pooled = false, pooled2 = false;
    if (graph_alloc(ctx, (void **)&rp, sizeof(uint64_t) * ((size_t)n + 1), &pooled) != cudaSuccess) {
        cudaGetLastError();
        return set_error(ctx, TC_ERR_OOM, "tc_build_csr: row_ptr allocation failed");
    }
    if (graph_alloc(ctx, (void **)&col, sizeof(uint32_t) * (size_t)(U + 1), &pooled2) != cudaSuccess) {
        cudaGetLastError();
        graph_free(ctx, rp, pooled);
        return set_error(ctx, TC_ERR_OOM, "tc_build_csr: col allocation failed");
    }
    *pooled_out = pooled;
    if (U) {
        k_compact<<<grid_for(nk, 256, cap), 256, 0, s>>>(cur, nk, flag, reinterpret_cast<const unsigned long long *>(pos),
                                                        col, src32);
        k_rowptr<<<grid_for(U + 1, 256, cap), 256, 0, s>>>(src32, U, n, rp);
    } else {
        k_empty_rowptr<<<grid_for((uint64_t)n + 1, 256, cap), 256, 0, s>>>(n, rp);
    }
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) {
        graph_free(ctx, rp, pooled);
        graph_free(ctx, col, pooled2);
        return cuda_error(ctx, e, "tc_build_csr kernels");
    }
    *rp_out = rp;
    *col_out = col;
    *slots_out = U;
    return max_degree_device(ctx, n, rp, max_deg);
}

tc_status validate_csr_device(tc_ctx *ctx, uint32_t n, const uint64_t *rp, const uint32_t *col, uint64_t slots,
                              int *ok) {
    cudaStream_t s = ctx->stream;
    const unsigned cap = (unsigned)ctx->num_sms * 16u;
    k_ctl_zero<<<1, 128, 0, s>>>(ctx->d_ctl);
    if (n) k_validate<<<grid_for((uint64_t)n * 32, 256, cap), 256, 0, s>>>(n, rp, col, slots, ctx->d_ctl);
    TC_CUDA(ctx, cudaGetLastError());
    tc_status st = pull(ctx);
    if (st != TC_OK) return st;
    *ok = ctx->h_ctl->error == 0 && (n > 0 || slots == 0);
    return TC_OK;
}

tc_status max_degree_device(tc_ctx *ctx, uint32_t n, const uint64_t *rp, uint32_t *max_deg) {
    cudaStream_t s = ctx->stream;
    const unsigned cap = (unsigned)ctx->num_sms * 16u;
    k_ctl_zero<<<1, 128, 0, s>>>(ctx->d_ctl);
    if (n) k_max_deg<<<grid_for(n, 256, cap), 256, 0, s>>>(n, rp, ctx->d_ctl);
    TC_CUDA(ctx, cudaGetLastError());
    tc_status st = pull(ctx);
    if (st != TC_OK) return st;
    *max_deg = ctx->h_ctl->max_s2;
    return TC_OK;
}

}  // namespace tc

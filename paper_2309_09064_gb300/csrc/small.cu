// small.cu -- plain counts of graphs of up to 65536 vertices, one or a disjoint
// union of many (tc_count_batch), under the degree order.
//
// The pairs are those of wedge.cu -- every triangle w, u < v found once, in the
// row N(v) of its latest vertex -- but taken from v's side: a warp marks N(v) in
// a bitmap over the graph's vertices (8 KB at most) and walks N(u) for every u in
// N(v), one bit test per neighbour.  That tries sum |N(u)| |{v}| pairs (two to
// three times the wedges) and needs nothing else: no ranks (a neighbour's degree
// and id say whether it precedes), no sorted rows, no entries, no tasks -- two
// kernels after the levels, where the tiles take eight.  Rows are kept as 16-bit
// ids relative to the graph's first vertex.
// The walk is bound by the ids' loads from L2 and the bit tests (shared memory).
// Measured (one GB300, whole call, before and after): against the tiles R-MAT 10
// 174 -> 104 us, R-MAT 13 of edge factor 16 266 -> 179 us, a uniform graph of
// 16384 vertices of mean degree 40 347 -> 212 us; against the classes of isect.cu
// 512 graphs of 64 .. 65536 vertices 13.5 -> 6.9 ms (this kernel 4.2).
#include <algorithm>

#include "pipeline.cuh"
#include "walk.cuh"

namespace tc {
namespace {

constexpr uint32_t kSmallMax = 65536;    // vertices of one graph (16-bit ids, degrees and levels)
constexpr uint32_t kLaneRow = 32;        // rows of degree <= 32: one lane each
constexpr uint32_t kBlockRow = 2048;     // rows of higher degree: a block each
constexpr uint32_t kSlice = 64;          // a row of more than this many u is walked by several warps
constexpr int kRowThreads = 256;
constexpr uint32_t kCountWarps = 8;      // of a block that walks rows
constexpr uint32_t kDirectBlocks = 128;  // grids of up to so many: every warp adds its sums itself
constexpr unsigned kGuardWatchdog = 0x80u;
constexpr long long kWatchdogCycles = 20000000000ll;  // about 10 s of SM clock

__device__ __forceinline__ uint32_t group_at(const GroupSpec &g, uint32_t x) {
    uint32_t a = 0, b = g.n_groups;
    while (b - a > 1) {
        const uint32_t m = (a + b) >> 1;
        if (g.vertex_start[m] <= x) a = m; else b = m;
    }
    return a;
}

// degree << 16 | level (modulo 2^16: levels are only compared across edges, where
// they differ by one at most)
__global__ void k_small_pack(uint32_t n, const uint32_t *__restrict__ deg, const uint32_t *__restrict__ L,
                             uint32_t *__restrict__ dl) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t x = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n; x += stride)
        dl[x] = deg[x] << 16 | (L[x] & 0xFFFFu);
}

struct SmallRows {
    uint16_t *ids;     // the rows: 16-byte units [(rp + 1) / 2, ...), as in wedge.cu
    uint2 *meta;       // by vertex: {first unit, |N| | level << 16}
    uint32_t *huge;    // rows a block fills
    uint2 *slices;     // {vertex, slice} of the rows walked by several warps
};

__device__ __forceinline__ void small_row_done(const SmallRows &o, uint32_t x, uint64_t b, uint32_t d, uint32_t level,
                                               Ctl *ctl) {
    o.meta[x] = make_uint2((uint32_t)((b + 1) >> 1), d | level << 16);
    if (d > kSlice) {
        const uint32_t k = (d + kSlice - 1) / kSlice, at = atomicAdd(&ctl->n_big, k);
        for (uint32_t i = 0; i < k; ++i) o.slices[at + i] = make_uint2(x, i);
    }
}

// N(x) of every vertex of degree <= kBlockRow, in CSR order, filled up to whole
// units with x's own id: whoever walks the row has x in its bitmap, so the count
// knows how often the padding is found (a vertex of degree >= 2 owns room for it,
// see wedge.cu; one of degree 1 closes no triangle and keeps an empty row).
__global__ void __launch_bounds__(kRowThreads) k_small_rows(uint32_t n, const uint64_t *__restrict__ rp,
                                                            const uint32_t *__restrict__ col,
                                                            const uint32_t *__restrict__ dl, GroupSpec groups,
                                                            SmallRows out,
                                                            uint32_t per_warp, Ctl *ctl) {
    const unsigned lane = lane_id();
    const unsigned lt = (1u << lane) - 1u;
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
        const uint32_t me = valid ? dl[x] : 0u;
        const uint32_t g = valid && groups.n_groups ? group_at(groups, (uint32_t)x) : 0u;
        const uint32_t base = groups.n_groups && valid ? groups.vertex_start[g] : 0u;
        if (valid && dx <= kLaneRow) {
            uint32_t d = 0;
            uint16_t *id = out.ids + 8 * ((b + 1) >> 1);
            for (uint32_t j0 = 0; j0 < dx; j0 += 8) {
                uint32_t y[8], q[8];
#pragma unroll
                for (uint32_t t = 0; t < 8; ++t) y[t] = j0 + t < dx ? col[b + j0 + t] : 0u;
#pragma unroll
                for (uint32_t t = 0; t < 8; ++t) q[t] = j0 + t < dx ? dl[y[t]] : 0u;
#pragma unroll
                for (uint32_t t = 0; t < 8; ++t) {
                    const uint32_t dy = q[t] >> 16;
                    if (!(j0 + t < dx && (dy > dx || (dy == dx && y[t] < (uint32_t)x)))) continue;
                    horizontal += ((q[t] ^ me) & 0xFFFFu) == 0;
                    if (dx >= 2) id[d++] = (uint16_t)(y[t] - base);
                }
            }
            for (uint32_t i = d; i & 7u; ++i) id[i] = (uint16_t)((uint32_t)x - base);
            small_row_done(out, (uint32_t)x, b, d, me & 0xFFFFu, ctl);
        }
        __syncwarp();
        if (valid && dx > kBlockRow) out.huge[atomicAdd(&ctl->n_huge, 1u)] = (uint32_t)x;
        unsigned pending = __ballot_sync(0xFFFFFFFFu, valid && dx > kLaneRow && dx <= kBlockRow);
        while (pending) {
            const int src = __ffs(pending) - 1;
            pending &= pending - 1;
            const uint32_t bx = c * per_warp + (uint32_t)src;
            const uint32_t bd = __shfl_sync(0xFFFFFFFFu, dx, src), bme = __shfl_sync(0xFFFFFFFFu, me, src);
            const uint32_t bbase = __shfl_sync(0xFFFFFFFFu, base, src);
            const uint64_t bb = __shfl_sync(0xFFFFFFFFu, b, src);
            uint16_t *id = out.ids + 8 * ((bb + 1) >> 1);
            uint32_t d = 0;
            for (uint32_t j0 = 0; j0 < bd; j0 += 128) {  // four neighbours per lane in flight
                uint32_t y[4], q[4];
#pragma unroll
                for (int t = 0; t < 4; ++t) y[t] = j0 + 32 * t + lane < bd ? col[bb + j0 + 32 * t + lane] : 0u;
#pragma unroll
                for (int t = 0; t < 4; ++t) q[t] = j0 + 32 * t + lane < bd ? dl[y[t]] : 0u;
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const uint32_t dy = q[t] >> 16;
                    const bool in = j0 + 32 * t + lane < bd && (dy > bd || (dy == bd && y[t] < bx));
                    const unsigned m = __ballot_sync(0xFFFFFFFFu, in);
                    if (in) {
                        id[d + __popc(m & lt)] = (uint16_t)(y[t] - bbase);
                        horizontal += ((q[t] ^ bme) & 0xFFFFu) == 0;
                    }
                    d += __popc(m);
                }
            }
            if (lane < ((0u - d) & 7u)) id[d + lane] = (uint16_t)(bx - bbase);
            if (lane == 0) small_row_done(out, bx, bb, d, bme & 0xFFFFu, ctl);
        }
    }
    horizontal = warp_sum(horizontal);
    if (lane == 0 && horizontal) atomicAdd(&ctl->e0, horizontal);
}

// Rows of degree above kBlockRow, a block each.
__global__ void __launch_bounds__(1024) k_small_rows_huge(const uint64_t *__restrict__ rp,
                                                          const uint32_t *__restrict__ col,
                                                          const uint32_t *__restrict__ dl, GroupSpec groups,
                                                          SmallRows out, Ctl *ctl) {
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
        const uint32_t x = out.huge[i];
        const uint64_t b = rp[x];
        const uint32_t dx = (uint32_t)(rp[x + 1] - b), me = dl[x];
        const uint32_t g = groups.n_groups ? group_at(groups, x) : 0u;
        const uint32_t base = groups.n_groups ? groups.vertex_start[g] : 0u;
        uint16_t *id = out.ids + 8 * ((b + 1) >> 1);
        uint32_t d = 0;
        for (uint32_t j0 = 0; j0 < dx; j0 += 4 * blockDim.x) {
            uint32_t y[4], q[4];
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
                q[t] = j < dx ? dl[y[t]] : 0u;
                const uint32_t dy = q[t] >> 16;
                m[t] = __ballot_sync(0xFFFFFFFFu, j < dx && (dy > dx || (dy == dx && y[t] < x)));
                mine += __popc(m[t]);
            }
            if (lane == 0) wcnt[warp] = mine;
            __syncthreads();
            const uint32_t v = wcnt[lane];
            uint32_t incl = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t z = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                if (lane >= (unsigned)o) incl += z;
            }
            uint32_t pos = d + __shfl_sync(0xFFFFFFFFu, incl - v, warp);
            d += __shfl_sync(0xFFFFFFFFu, incl, 31);
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                if ((m[t] >> lane) & 1u) {
                    id[pos + __popc(m[t] & lt)] = (uint16_t)(y[t] - base);
                    horizontal += ((q[t] ^ me) & 0xFFFFu) == 0;
                }
                pos += __popc(m[t]);
            }
            __syncthreads();
        }
        if (threadIdx.x < ((0u - d) & 7u)) id[d + threadIdx.x] = (uint16_t)(x - base);
        if (threadIdx.x == 0) small_row_done(out, x, b, d, me & 0xFFFFu, ctl);
    }
    horizontal = warp_sum(horizontal);
    if (lane == 0 && horizontal) atomicAdd(&ctl->e0, horizontal);
}

// The pairs of every row: slices of the long ones first, then the others in
// chunks of per_warp.  A warp's bitmap holds N(v) (with kSplit, in pairs of words:
// the second has N(v)'s horizontal members, so a hit beside a horizontal u-v edge
// is split without looking w up); eight groups of four lanes walk the rows of 32
// u at a time, 32 ids (64 bytes) a step, the next step's ids loaded ahead.
// !kSplit credits every graph's triangles to groups.counts.
template <bool kSplit>
__global__ void __launch_bounds__(512) k_small_count(uint32_t n, const uint16_t *__restrict__ ids,
                                                     const uint2 *__restrict__ meta,
                                                     const uint2 *__restrict__ slices, GroupSpec groups,
                                                     uint32_t words, uint32_t per_warp, Ctl *ctl) {
    extern __shared__ __align__(16) uint32_t smem[];
    __shared__ volatile unsigned long long s_sum[kCountWarps][5];  // {same, cross, probes, marked, walks}
    __shared__ unsigned int s_done;
    if (ctl->e0 == 0) return;  // (every triangle has a horizontal edge)
    if (gridDim.x > kDirectBlocks) {
        if (threadIdx.x == 0) s_done = 0;
        __syncthreads();
    }
    constexpr uint32_t kW = kSplit ? 2 : 1;
    const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
    const uint32_t sub = lane & 3u;
    uint32_t *map = smem + warp * (kW * words + 128);
    uint4 *ent = reinterpret_cast<uint4 *>(map + kW * words);
    const uint4 *unit = reinterpret_cast<const uint4 *>(ids);
    for (uint32_t i = lane; i < kW * words; i += 32) map[i] = 0;
    __syncwarp();
    unsigned long long same = 0, cross = 0, probes = 0, group_sum = 0;
    unsigned long long marked = 0;  // ids put into the bitmap by this lane
    uint32_t walks = 0;
    uint32_t group = 0, base = 0, group_end = groups.n_groups ? 0u : 0xFFFFFFFFu;  // group_end 0: none yet
    const long long t_start = clock64();
    // pairs of v with u among the keys [lo, hi) of its row
    auto walk = [&](uint32_t v, uint32_t lo, uint32_t hi) {
        if (groups.n_groups && (v >= group_end || v < base)) {  // (the warp's current group)
            const unsigned long long s = warp_sum(group_sum);
            if (lane == 0 && s) atomicAdd(&groups.counts[group], s);
            group_sum = 0;
            group = group_at(groups, v);
            base = groups.vertex_start[group];
            group_end = groups.vertex_start[group + 1];
        }
        const uint2 mv = meta[v];
        const uint32_t d = mv.y & 0xFFFFu, level = mv.y >> 16;
        const uint16_t *row = ids + 8ull * mv.x;
        ++walks;
        for (uint32_t i = lane; i < d; i += 32) {
            ++marked;
            const uint32_t e = row[i], bit = 1u << (e & 31u);
            atomicOr(&map[kW * (e >> 5)], bit);
            if (kSplit && meta[base + e].y >> 16 == level) atomicOr(&map[kW * (e >> 5) + 1], bit);
        }
        __syncwarp();
        uint32_t tot = 0, sam = 0;
        for (uint32_t j0 = lo; j0 < hi; j0 += 32) {
            uint2 m = make_uint2(0, 0);
            if (j0 + lane < hi) m = meta[base + row[j0 + lane]];
            const uint32_t len = m.y & 0xFFFFu, units = (len + 7) / 8;
            probes += len;
            tot -= 8 * units - len;  // the padding is u itself, which v's bitmap has
            if (kSplit && m.y >> 16 == level) sam -= 8 * units - len;
            __syncwarp();
            ent[lane] = make_uint4(m.x, units, m.y >> 16 == level, 0u);
            __syncwarp();
            Walk w = share_steps((units + 3) / 4);
            uint4 cur = ent[w.i];
            uint32_t at = cur.x + sub + 4 * w.skip;
            int rem = (int)cur.y - (int)(4 * w.skip + sub);
            // ids of the group's next step; past its end none
            auto fetch = [&](uint4 &q, bool &on, uint32_t &flag) {
                on = false;
                if (w.left) {
                    --w.left;
                    while (rem + (int)sub <= 0) {
                        w.i = (w.i + 1) & 31u;
                        cur = ent[w.i];
                        at = cur.x + sub;
                        rem = (int)cur.y - (int)sub;
                    }
                    if (rem > 0) {
                        q = __ldg(unit + at);
                        on = true;
                    }
                    at += 4;
                    rem -= 4;
                }
                flag = cur.z;
            };
            auto look = [&](uint32_t e, uint32_t flag) {
                if constexpr (kSplit) {
                    const uint2 x = reinterpret_cast<const uint2 *>(map)[e >> 5];
                    tot += (x.x >> (e & 31u)) & 1u;
                    sam += (x.y >> (e & 31u)) & flag;
                } else {
                    tot += (map[e >> 5] >> (e & 31u)) & 1u;
                }
            };
            uint4 a = make_uint4(0, 0, 0, 0), a1 = a;
            bool on, on1;
            uint32_t flag, flag1;
            fetch(a, on, flag);
            for (uint32_t k = 0; k < w.iters; ++k) {
                fetch(a1, on1, flag1);
                if (on) {
                    look(a.x & 0xFFFFu, flag);
                    look(a.x >> 16, flag);
                    look(a.y & 0xFFFFu, flag);
                    look(a.y >> 16, flag);
                    look(a.z & 0xFFFFu, flag);
                    look(a.z >> 16, flag);
                    look(a.w & 0xFFFFu, flag);
                    look(a.w >> 16, flag);
                }
                a = a1;
                on = on1;
                flag = flag1;
            }
        }
        __syncwarp();
        for (uint32_t i = lane; i < d; i += 32) {
            const uint32_t e = row[i];
            map[kW * (e >> 5)] = 0;
            if (kSplit) map[kW * (e >> 5) + 1] = 0;
        }
        __syncwarp();
        // (a lane's share can be negative: the padding was taken off by the lane that fetched u's place)
        same += (unsigned long long)(long long)(int)sam;
        cross += (unsigned long long)(long long)(int)(tot - sam);
        group_sum += (unsigned long long)(long long)(int)tot;
    };
    auto expired = [&] {
        if (clock64() - t_start <= kWatchdogCycles) return false;
        if (lane == 0) atomicOr(&ctl->error, kGuardWatchdog);
        return true;
    };
    const uint32_t ns = ctl->n_big;
    for (;;) {  // one slice of a long row
        uint32_t i = 0;
        if (lane == 0) i = atomicAdd(&ctl->task_next[1], 1u);
        i = __shfl_sync(0xFFFFFFFFu, i, 0);
        if (i >= ns || __any_sync(0xFFFFFFFFu, expired())) break;
        const uint2 t = slices[i];
        const uint32_t d = meta[t.x].y & 0xFFFFu;
        walk(t.x, t.y * kSlice, min(d, (t.y + 1) * kSlice));
    }
    const uint64_t chunks = ((uint64_t)n + per_warp - 1) / per_warp;
    for (;;) {
        unsigned int c = 0;
        if (lane == 0) c = atomicAdd(&ctl->task_next[0], 1u);
        c = __shfl_sync(0xFFFFFFFFu, c, 0);
        if (c >= chunks || __any_sync(0xFFFFFFFFu, expired())) break;
        const uint64_t x = (uint64_t)c * per_warp + lane;
        const uint32_t d = lane < per_warp && x < n ? meta[x].y & 0xFFFFu : 0u;
        unsigned pending = __ballot_sync(0xFFFFFFFFu, d >= 2 && d <= kSlice);
        while (pending) {
            const int src = __ffs(pending) - 1;
            pending &= pending - 1;
            walk(c * per_warp + (uint32_t)src, 0, __shfl_sync(0xFFFFFFFFu, d, src));
        }
    }
    if (groups.n_groups) {
        const unsigned long long s = warp_sum(group_sum);
        if (lane == 0 && s) atomicAdd(&groups.counts[group], s);
    }
    same = warp_sum(same);
    cross = warp_sum(cross);
    probes = warp_sum(probes);
    marked = warp_sum(marked);
    unsigned long long *const to = lane == 0   ? &ctl->t_same
                                   : lane == 1 ? &ctl->t_cross
                                   : lane == 2 ? &ctl->cls_probes[0]
                                   : lane == 3 ? &ctl->cls_build[0]
                                               : &ctl->cls_rows[0];
    unsigned long long sum = lane == 0 ? same : lane == 1 ? cross : lane == 2 ? probes : lane == 3 ? marked : walks;
    // In larger grids the block's last warp adds its warps' sums up: the warps' own atomics, on the same few
    // addresses, take 10 us of a graph of 20000 vertices.  (At 1024 vertices the reduction takes 1 us more.)
    if (gridDim.x > kDirectBlocks) {
        bool last = false;
        if (lane < 5) s_sum[warp][lane] = sum;
        __syncwarp();
        if (lane == 0) {
            __threadfence_block();
            last = atomicAdd(&s_done, 1u) + 1 == blockDim.x / 32;
        }
        if (!__shfl_sync(0xFFFFFFFFu, last, 0)) return;
        __threadfence_block();
        sum = 0;
        for (uint32_t w = 0; lane < 5 && w < blockDim.x / 32; ++w) sum += s_sum[w][lane];
    }
    if (lane < 5 && sum) atomicAdd(to, sum);
}

unsigned grid_for(uint64_t work, unsigned threads, unsigned cap) {
    uint64_t b = (work + threads - 1) / threads;
    if (b < 1) b = 1;
    if (b > cap) b = cap;
    return (unsigned)b;
}

}  // namespace

// One graph, or a union whose largest has max_n vertices.  A tile's lookup serves
// 32 u's and a bitmap's one, so graphs of high mean degree take the tiles, and a
// single large one too (both sides are measured at kSmallOne).
bool small_path(const tc_ctx *ctx, uint32_t n, uint64_t slots, uint32_t max_deg, const GroupSpec &groups) {
    const uint32_t max_n = groups.n_groups ? groups.max_n : n;
    return wedge_path(ctx, n, slots, max_deg) && max_n <= (groups.n_groups ? kSmallMax : kSmallOne) &&
           slots <= 64ull * n;
}

tc_status small_count(tc_ctx *ctx, const PipeBufs &b, uint32_t n, uint32_t max_deg) {
    cudaStream_t s = ctx->stream;
    const unsigned cap = (unsigned)ctx->num_sms * 16u;
    const bool grouped = b.groups.n_groups != 0;
    const uint32_t per_warp = n >= (1u << 18) ? 32u : n >= (1u << 15) ? 8u : 2u;
    SmallRows rows{reinterpret_cast<uint16_t *>(b.erec), b.lv, b.huge, b.task_pool};
    uint32_t *dl = b.rank;
    k_small_pack<<<grid_for(n, 256, cap), 256, 0, s>>>(n, b.deg, b.L, dl);
    k_small_rows<<<grid_for((uint64_t)n * (32 / per_warp), kRowThreads, cap), kRowThreads, 0, s>>>(
        n, b.rp, b.col, dl, b.groups, rows, per_warp, ctx->d_ctl);
    if (max_deg > kBlockRow)
        k_small_rows_huge<<<(unsigned)ctx->num_sms, 1024, 0, s>>>(b.rp, b.col, dl, b.groups, rows, ctx->d_ctl);
    note_launch(ctx, max_deg > kBlockRow ? 4 : 3);
    TC_CUDA(ctx, cudaEventRecord(ctx->ev[2], s));
    TC_CUDA(ctx, cudaEventRecord(ctx->ev[4], s));
    const uint32_t words = ((grouped ? b.groups.max_n : n) + 127) / 128 * 4;  // whole 16-byte pieces
    const size_t per = 4ull * ((grouped ? 1 : 2) * words + 128);
    const uint32_t warps = (uint32_t)std::min<size_t>(kCountWarps, kSmemLimitBytes / per);
    const size_t smem = per * warps;
    auto kern = grouped ? k_small_count<false> : k_small_count<true>;
    TC_CUDA(ctx, allow_dynamic_smem((const void *)kern));
    int per_sm = 0;
    TC_CUDA(ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32 * warps, smem));
    const uint64_t blocks = ((uint64_t)n + per_warp * warps - 1) / (per_warp * warps);
    kern<<<(unsigned)std::min<uint64_t>(blocks, (uint64_t)ctx->num_sms * std::max(per_sm, 1)), 32 * warps, smem, s>>>(
        n, rows.ids, rows.meta, rows.slices, b.groups, words, per_warp, ctx->d_ctl);
    TC_CUDA(ctx, cudaEventRecord(ctx->ev[5], s));
    ctx->isect_flags = 1u;
    TC_CUDA(ctx, cudaGetLastError());
    return TC_OK;
}

}  // namespace tc

// warp_sort.cuh -- sorting up to 1024 32-bit keys in shared memory with one warp.
#pragma once

#include "tc_internal.cuh"

namespace tc {

// Ascending bitonic sort of 32 * E keys by one warp, E consecutive ones per
// lane in registers: compares across lanes are shuffles, the others stay in
// the lane (in shared memory every compare costs two loads and two stores).
template <int E>
__device__ __forceinline__ void lane_sort(uint32_t (&v)[E]) {
    const unsigned lane = lane_id();
#pragma unroll
    for (int k = 2; k <= 32 * E; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            if (j >= E) {
                const bool low = ((lane & (j / E)) == 0) == (((lane * E) & k) == 0);
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const uint32_t o = __shfl_xor_sync(0xFFFFFFFFu, v[e], j / E);
                    v[e] = low ? min(v[e], o) : max(v[e], o);
                }
            } else {
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    if (e & j) continue;
                    const bool up = k < E ? (e & k) == 0 : ((lane * E) & k) == 0;
                    const uint32_t x = v[e], y = v[e | j];
                    v[e] = up ? min(x, y) : max(x, y);
                    v[e | j] = up ? max(x, y) : min(x, y);
                }
            }
        }
    }
}

// Sort buf[0..d), d <= 32 * E, in place (descending: written back reversed).
template <int E>
__device__ __forceinline__ void warp_sort(uint32_t *buf, uint32_t d, bool descending = false) {
    const unsigned lane = lane_id();
    uint32_t v[E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
        v[e] = e * 32 + lane < d ? buf[e * 32 + lane] : kEmpty;
        if (descending) v[e] = ~v[e];
    }
    lane_sort<E>(v);
    __syncwarp();
#pragma unroll
    for (int e = 0; e < E; ++e)
        if (descending) v[e] = ~v[e];
    if constexpr (E % 4 == 0) {
#pragma unroll
        for (int e = 0; e < E; e += 4)
            reinterpret_cast<uint4 *>(buf)[(lane * E + e) / 4] = make_uint4(v[e], v[e + 1], v[e + 2], v[e + 3]);
    } else {
#pragma unroll
        for (int e = 0; e < E; ++e) buf[lane * E + e] = v[e];
    }
    __syncwarp();
}

// The last log2(256) steps of a bitonic merge: buf[0..256) bitonic -> sorted.
__device__ __forceinline__ void warp_merge_256(uint32_t *buf, bool descending) {
    constexpr int E = 8;
    const unsigned lane = lane_id();
    uint32_t v[E];
#pragma unroll
    for (int e = 0; e < E; e += 4) {
        const uint4 q = reinterpret_cast<const uint4 *>(buf)[(lane * E + e) / 4];
        v[e] = q.x, v[e + 1] = q.y, v[e + 2] = q.z, v[e + 3] = q.w;
    }
    if (descending) {
#pragma unroll
        for (int e = 0; e < E; ++e) v[e] = ~v[e];
    }
#pragma unroll
    for (int j = 128; j > 0; j >>= 1) {
        if (j >= E) {
            const bool low = (lane & (j / E)) == 0;
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const uint32_t o = __shfl_xor_sync(0xFFFFFFFFu, v[e], j / E);
                v[e] = low ? min(v[e], o) : max(v[e], o);
            }
        } else {
#pragma unroll
            for (int e = 0; e < E; ++e) {
                if (e & j) continue;
                const uint32_t x = v[e], y = v[e | j];
                v[e] = min(x, y);
                v[e | j] = max(x, y);
            }
        }
    }
    if (descending) {
#pragma unroll
        for (int e = 0; e < E; ++e) v[e] = ~v[e];
    }
#pragma unroll
    for (int e = 0; e < E; e += 4)
        reinterpret_cast<uint4 *>(buf)[(lane * E + e) / 4] = make_uint4(v[e], v[e + 1], v[e + 2], v[e + 3]);
    __syncwarp();
}

// Sort buf[0..d), 256 < d <= P (512 or 1024, kEmpty from d on): runs of 256 in
// registers, their merges' first steps in shared memory.  (One register sort of
// 1024 keys is 3500 instructions; two of them beside the smaller ones miss the
// instruction cache.)
__device__ __forceinline__ void warp_sort_large(uint32_t *buf, uint32_t d, uint32_t P) {
    const unsigned lane = lane_id();
    for (uint32_t c = 0; c < P; c += 256) warp_sort<8>(buf + c, d > c ? d - c : 0u, (c & 256u) != 0);
    for (uint32_t k = 512; k <= P; k <<= 1) {
        for (uint32_t j = k >> 1; j >= 256; j >>= 1) {
            for (uint32_t p = lane; p < P / 2; p += 32) {
                const uint32_t i = ((p & ~(j - 1)) << 1) | (p & (j - 1)), l = i | j;
                const uint32_t a = buf[i], c = buf[l];
                if ((a > c) == ((i & k) == 0)) {
                    buf[i] = c;
                    buf[l] = a;
                }
            }
            __syncwarp();
        }
        for (uint32_t c = 0; c < P; c += 256) warp_merge_256(buf + c, (c & k) != 0);
    }
}

// Sort buf[0..d), d <= 1024 (the buffer holds 1024 words).
__device__ __forceinline__ void warp_sort_any(uint32_t *buf, uint32_t d) {
    if (d <= 32) warp_sort<1>(buf, d);
    else if (d <= 64) warp_sort<2>(buf, d);
    else if (d <= 128) warp_sort<4>(buf, d);
    else if (d <= 256) warp_sort<8>(buf, d);
    else warp_sort_large(buf, d, d <= 512 ? 512u : 1024u);
}

}  // namespace tc

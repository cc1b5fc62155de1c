// kd_block_sort.cuh -- radix sorting inside one thread block.
#pragma once

#include "kd_internal.cuh"

namespace kd {

// One stable 8-bit LSD pass over the block's n elements, E rows of 32 per
// warp: the element at place warp * 32 E + e * 32 + lane is (key[e], id[e]);
// on return the arrays hold the new order and are reloaded from it.  Lanes
// of equal digits are found by a ballot per digit bit (the match
// instruction's cost grows with the distinct digits in a warp).
template <int NW, int E>
__device__ __forceinline__ void block_pass(uint32_t (&key)[E], uint32_t (&id)[E], int shift, int n, uint32_t* s_key,
                                           uint16_t* s_idx, uint16_t (*wc)[RADIX], uint32_t* s_ws) {
    constexpr int Q = NW / 8;  // threads per digit of the scan, each over 8 warps
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t lt = lanemask_lt();
    reinterpret_cast<uint4*>(wc[warp])[lane] = make_uint4(0, 0, 0, 0);
    __syncwarp();
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const bool in = warp * 32 * E + e * 32 + lane < n;
        const uint32_t d = (key[e] >> shift) & 255u;
        uint32_t peers = __ballot_sync(0xffffffffu, in);
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            const uint32_t v = __ballot_sync(0xffffffffu, (d >> b) & 1u);
            peers &= (d >> b) & 1u ? v : ~v;
        }
        const uint32_t base = wc[warp][d];
        id[e] |= (base + __popc(peers & lt)) << 16;  // the rank rides with the index (14 bits)
        __syncwarp();
        if (in && lane == 31 - __clz(peers)) wc[warp][d] = (uint16_t)(base + __popc(peers));
        __syncwarp();
    }
    __syncthreads();
    {
        const int d = tid / Q, w0 = tid % Q * 8;
        uint32_t c[8], sum = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            c[i] = wc[w0 + i][d];
            sum += c[i];
        }
        uint32_t incl = sum;
#pragma unroll
        for (int o = 1; o < Q; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (tid % Q >= o) incl += y;
        }
        const uint32_t total = __shfl_sync(0xffffffffu, incl, lane | (Q - 1));  // of digit d
        uint32_t x = total;
#pragma unroll
        for (int o = Q; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) s_ws[warp] = x;
        __syncthreads();
        uint32_t run = __reduce_add_sync(0xffffffffu, lane < warp ? s_ws[lane] : 0u) + x - total + incl - sum;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            wc[w0 + i][d] = (uint16_t)run;
            run += c[i];
        }
    }
    __syncthreads();
#pragma unroll
    for (int e = 0; e < E; ++e) {
        if (warp * 32 * E + e * 32 + lane < n) {
            const uint32_t p = wc[warp][(key[e] >> shift) & 255u] + (id[e] >> 16);
            s_key[p] = key[e];
            s_idx[p] = (uint16_t)id[e];
        }
    }
    __syncthreads();
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int o = warp * 32 * E + e * 32 + lane;
        key[e] = o < n ? s_key[o] : 0u;
        id[e] = o < n ? s_idx[o] : 0u;
    }
}

// The block's sort word of a coordinate: the BITS bits of its key from the
// highest one in which the elements differ (those above are common).
// Elements of equal words keep their order and are left to the caller, who
// finds few of them while BITS is well above the logarithm of their number.
template <int BITS, typename KW>
__device__ __forceinline__ int word_shift(KW diff) {
    const int high = sizeof(KW) == 8 ? 63 - __clzll((long long)diff) : 31 - __clz((int)(uint32_t)diff);
    return high >= BITS ? high - BITS + 1 : 0;
}
template <int BITS, typename KW>
__device__ __forceinline__ uint32_t sort_word(KW key, int shift) {
    return (uint32_t)(key >> shift) & (uint32_t)((1ull << BITS) - 1);
}

// AND and OR of the block's keys, from each thread's: the bits that differ.
// s_w: 4 words (set by the call, free after the next barrier).  All threads.
template <typename KW>
__device__ __forceinline__ KW block_diff(KW a, KW r, uint32_t* s_w) {
    const int lane = threadIdx.x & 31;
    if (threadIdx.x < 4) s_w[threadIdx.x] = threadIdx.x < 2 ? 0xffffffffu : 0u;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < (int)sizeof(KW) / 4; ++w) {
        const uint32_t aw = __reduce_and_sync(0xffffffffu, (uint32_t)((uint64_t)a >> (32 * w)));
        const uint32_t rw = __reduce_or_sync(0xffffffffu, (uint32_t)((uint64_t)r >> (32 * w)));
        if (lane == 0) {
            atomicAnd(&s_w[w], aw);
            atomicOr(&s_w[2 + w], rw);
        }
    }
    __syncthreads();
    if constexpr (sizeof(KW) == 8)
        return (KW)(((uint64_t)(s_w[1] ^ s_w[3]) << 32) | (s_w[0] ^ s_w[2]));
    else
        return (KW)(s_w[0] ^ s_w[2]);
}

}  // namespace kd

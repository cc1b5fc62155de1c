// kd_small.cu -- presort of a small cloud, one thread block per super key.
//
// Section 2.1's presort (k index arrays sorted by the cyclic super keys,
// duplicate tuples removed) for clouds of at most SMALL_MAX tuples, where a
// sort pass over the whole GPU is all launch latency:
//   k_small_sort  block d sorts the tuple indices by super key d in shared
//                 memory and removes duplicates;
//   k_small_recs  the rank records the build reads, from the arrays and
//                 their inverses;
//   k_small_keys  the key planes in array-0 order (median-selection build).
// kd_presort_noalloc is the first of them alone.
#include <cstdint>

#include "kd_block_sort.cuh"

namespace kd {

constexpr int SMALL_MAX = 16384;
constexpr int SMALL_RUN = 32;  // longest run of equal x_d ordered by compares

// Key of a coordinate (floats are checked for NaN before).
template <typename T>
__device__ __forceinline__ auto small_key(T v) {
    int nan = 0;
    return key_of(v, &nan);
}

template <typename KW, int NW, int E>
constexpr size_t small_smem() {
    return (size_t)32 * NW * E * (sizeof(KW) + 2);
}

// Outputs of k_small_sort: row d of arr (stride arr_stride) gets the
// deduplicated super-key-d order, row d of inv (optional) the place of every
// kept tuple in it; m the number of kept tuples, as 64 bits, or as 32 bits
// with KD_ENAN (-6) for a NaN coordinate; err the error bits.
struct SmallOut {
    uint32_t *arr, *inv;
    int64_t arr_stride, inv_stride;
    int64_t* m64;
    int32_t* m32;
    int* err;
};

// Block d: the indices of n tuples (at most 32 NW E) by super key d.  First a
// stable radix sort by the leading bits of x_d (16, or 24 above 2048
// tuples); then runs of equal words are ordered by the super key and the
// index by compares, or, where a run exceeds SMALL_RUN, everything is sorted
// again by the whole super key, least significant coordinate first, over
// the bytes that differ.  Bound by shared-memory latency and issue on its
// one SM; 16384 float32 tuples of k = 3: 83 us for the three arrays (a bitonic
// sort with super-key compares took 284).
template <typename T, typename KW, int NW, int E>
__global__ void __launch_bounds__(32 * NW, 1) k_small_sort(const T* __restrict__ coords, int n, int k,
                                                           const SmallOut out) {
    constexpr int NT = 32 * NW;
    extern __shared__ __align__(16) unsigned char ssm[];
    uint32_t* s_key = reinterpret_cast<uint32_t*>(ssm);                       // the word being sorted ...
    KW* s_full = reinterpret_cast<KW*>(ssm);                                  // ... then x_d in its order
    uint16_t* s_idx = reinterpret_cast<uint16_t*>(ssm + sizeof(KW) * NT * E);
    __shared__ __align__(16) uint16_t wc[NW][RADIX];
    __shared__ uint32_t s_ws[32], s_w[4];
    constexpr int BITS = NT * E <= 2048 ? 16 : 24;
    const int d = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int base = warp * 32 * E + lane;  // place of row 0's element
    if constexpr (sizeof(T) == 4 && T(0.5) != T(0)) {  // floats
        bool nan = false;
        for (int i = tid; i < n * k; i += NT) nan |= coords[i] != coords[i];
        if (__syncthreads_or(nan)) {
            if (d == 0 && tid == 0) {
                if (out.err) atomicOr(out.err, ERR_NAN);
                if (out.m32) *out.m32 = -6;
            }
            return;
        }
    }
    uint32_t key[E], id[E];
    // loads the current order (identity: the input's) and returns the bits in
    // which its x_c differ
    auto load = [&](int c, bool identity) {
        KW a = ~(KW)0, r = 0;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int o = base + e * 32;
            id[e] = identity ? (uint32_t)o : (o < n ? s_idx[o] : 0u);
            if (o < n) {
                const KW x = small_key(coords[(int64_t)id[e] * k + c]);
                a &= x;
                r |= x;
                if (identity) s_idx[o] = (uint16_t)o;
            }
        }
        return block_diff(a, r, s_w);
    };
    // key[]: bits from `shift` up of the elements' x_c
    auto words = [&](int c, int shift) {
#pragma unroll
        for (int e = 0; e < E; ++e)
            key[e] = base + e * 32 < n ? (uint32_t)(small_key(coords[(int64_t)id[e] * k + c]) >> shift) : 0u;
    };
    // stable sort of the current order by the whole of x_c
    auto sort_by = [&](int c, bool identity) {
        const KW differ = load(c, identity);
        __syncthreads();
#pragma unroll
        for (int w = 0; w < (int)sizeof(KW) * 8; w += 32) {
            if ((uint32_t)(differ >> w) == 0) continue;
            words(c, w);
            for (int b = 0; b < 32; b += 8)
                if (((uint32_t)(differ >> w) >> b) & 255u) block_pass<NW, E>(key, id, b, n, s_key, s_idx, wc, s_ws);
        }
    };
    auto fill_keys = [&]() {  // s_full: x_d in the current order
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int o = base + e * 32;
            if (o < n) s_full[o] = small_key(coords[(int64_t)s_idx[o] * k + d]);
        }
        __syncthreads();
    };
    // tuple i before tuple j by super key d and the index
    auto before = [&](int i, int j) {
        for (int r = 0; r < k; ++r) {
            const int c = d + r < k ? d + r : d + r - k;
            const KW x = small_key(coords[(int64_t)i * k + c]), y = small_key(coords[(int64_t)j * k + c]);
            if (x != y) return x < y;
        }
        return i < j;
    };
    const KW differ = load(d, true);
    const int shift = word_shift<BITS>(differ);
    if (differ != 0) {
        words(d, shift);
#pragma unroll
        for (int e = 0; e < E; ++e) key[e] &= (1u << BITS) - 1u;
        for (int b = 0; b < BITS; b += 8) block_pass<NW, E>(key, id, b, n, s_key, s_idx, wc, s_ws);
    }
    __syncthreads();
    fill_keys();
    auto word = [&](int o) { return sort_word<BITS>(s_full[o], shift); };
    {
        bool tie = false, lng = false;
        for (int e = 0; e < E; ++e) {
            const int o = base + e * 32;
            if (o + 1 >= n || word(o + 1) != word(o)) continue;
            tie = true;
            lng |= o + SMALL_RUN < n && word(o + SMALL_RUN) == word(o);
        }
        if (__syncthreads_or(lng)) {
            for (int r = k - 1; r >= 0; --r) {
                sort_by(d + r < k ? d + r : d + r - k, r == k - 1);
                __syncthreads();
            }
            fill_keys();
        } else if (__syncthreads_or(tie)) {
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const int o = base + e * 32;
                id[e] = 0;
                key[e] = 0xffffffffu;  // the element's new place, if it is in a run
                if (o >= n) continue;
                const uint32_t x = word(o);
                int s = o, f = o;
                while (s > 0 && word(s - 1) == x) --s;
                while (f + 1 < n && word(f + 1) == x) ++f;
                if (s == f) continue;
                id[e] = s_idx[o];
                int c = s;
                for (int j = s; j <= f; ++j) c += j != o && before(s_idx[j], (int)id[e]) ? 1 : 0;
                key[e] = (uint32_t)c;
            }
            __syncthreads();
#pragma unroll
            for (int e = 0; e < E; ++e)
                if (key[e] != 0xffffffffu) s_idx[key[e]] = (uint16_t)id[e];
            __syncthreads();
            fill_keys();
        }
    }
    // a tuple equal to its predecessor goes (the smallest index comes first)
    uint32_t keep[E], cnt = 0;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int o = base + e * 32;
        bool kp = o < n;
        if (kp && o > 0 && s_full[o - 1] == s_full[o]) {
            const int i = s_idx[o - 1], j = s_idx[o];
            bool same = true;
            for (int c = 0; c < k && same; ++c)
                same = small_key(coords[(int64_t)i * k + c]) == small_key(coords[(int64_t)j * k + c]);
            kp = !same;
        }
        keep[e] = __ballot_sync(0xffffffffu, kp);
        cnt += __popc(keep[e]);
    }
    if (lane == 0) s_ws[warp] = cnt;
    __syncthreads();
    uint32_t pos = __reduce_add_sync(0xffffffffu, lane < warp ? s_ws[lane] : 0u);
    if (d == 0 && tid == NT - 1) {
        if (out.m64) *out.m64 = pos + cnt;
        if (out.m32) *out.m32 = (int32_t)(pos + cnt);
    }
    uint32_t* arr = out.arr + d * out.arr_stride;
    uint32_t* inv = out.inv ? out.inv + d * out.inv_stride : nullptr;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        if ((keep[e] >> lane) & 1u) {
            const uint32_t p = pos + __popc(keep[e] & lanemask_lt());
            const uint32_t t = s_idx[base + e * 32];
            arr[p] = t;
            if (inv) inv[t] = p;
        }
        pos += __popc(keep[e]);
    }
}

// rec[d][p][i] = place in array p of the tuple at place i of array d (p != d;
// array 0 also its own places), and perm0 = array 0.  Block row y: array d.
__global__ void __launch_bounds__(256) k_small_recs(const int64_t* __restrict__ m_ptr, int k,
                                                    const uint32_t* __restrict__ arr, const uint32_t* __restrict__ inv,
                                                    int64_t stride, const __grid_constant__ AllPlanes rec,
                                                    uint32_t* __restrict__ perm0) {
    const int i = blockIdx.x * 256 + threadIdx.x, d = blockIdx.y;
    if (i >= *m_ptr) return;
    const uint32_t t = arr[d * stride + i];
    if (d == 0) perm0[i] = t;
    if (k < 2) return;
    for (int p = 0; p < k; ++p)
        if (p != d) rec.p[d][p][i] = inv[p * stride + t];
    if (d == 0) rec.p[0][0][i] = (uint32_t)i;
}

// Key planes (stride words apart) of the tuples in array-0 order.
template <typename T, typename KW>
__global__ void __launch_bounds__(256) k_small_keys(const int64_t* __restrict__ m_ptr, int k,
                                                    const T* __restrict__ coords, const uint32_t* __restrict__ perm0,
                                                    KW* __restrict__ keys, int64_t stride) {
    const int i = blockIdx.x * 256 + threadIdx.x;
    if (i >= *m_ptr) return;
    const int64_t t = perm0[i];
    for (int d = 0; d < k; ++d) keys[d * stride + i] = small_key(coords[t * k + d]);
}

// ------------------------------------------------------------ launchers
int small_presort_max() { return SMALL_MAX; }

template <typename T, typename KW, int NW, int E>
static cudaError_t small_sort_as(const void* coords, int n, int k, int narrays, const SmallOut& out, cudaStream_t s) {
    // (the error of the launch call itself: one pending from earlier work is neither reported nor cleared)
    const T* c = static_cast<const T*>(coords);
    SmallOut o = out;
    void* argv[] = {&c, &n, &k, &o};
    return cudaLaunchKernel(reinterpret_cast<const void*>(&k_small_sort<T, KW, NW, E>), dim3(narrays), dim3(32 * NW),
                            argv, small_smem<KW, NW, E>(), s);
}

// The fewest rows that hold n: a block of 8 warps up to 1024 tuples (its
// barriers and scans are shorter), of 32 warps above.
template <typename T, typename KW>
static cudaError_t small_sort_of(const void* coords, int n, int k, int narrays, const SmallOut& out, cudaStream_t s) {
    if (n <= 256) return small_sort_as<T, KW, 8, 1>(coords, n, k, narrays, out, s);
    if (n <= 1024) return small_sort_as<T, KW, 8, 4>(coords, n, k, narrays, out, s);
    if (n <= 2048) return small_sort_as<T, KW, 32, 2>(coords, n, k, narrays, out, s);
    if (n <= 4096) return small_sort_as<T, KW, 32, 4>(coords, n, k, narrays, out, s);
    if (n <= 8192) return small_sort_as<T, KW, 32, 8>(coords, n, k, narrays, out, s);
    return small_sort_as<T, KW, 32, 16>(coords, n, k, narrays, out, s);
}

static cudaError_t small_sort(int dtype, const void* coords, int n, int k, int narrays, const SmallOut& out,
                              cudaStream_t s) {
    if (n < 1 || n > SMALL_MAX) return cudaErrorInvalidValue;
    if (dtype == 0) return small_sort_of<int32_t, uint32_t>(coords, n, k, narrays, out, s);
    if (dtype == 1) return small_sort_of<int64_t, uint64_t>(coords, n, k, narrays, out, s);
    return small_sort_of<float, uint32_t>(coords, n, k, narrays, out, s);
}

// kd_presort_noalloc: rows of n in out, m (or KD_ENAN) in m_out.
cudaError_t launch_small_arrays(int dtype, const void* coords, int n, int k, int32_t* rows, int32_t* m_out,
                                cudaStream_t s) {
    SmallOut o{};
    o.arr = reinterpret_cast<uint32_t*>(rows);
    o.arr_stride = n;
    o.m32 = m_out;
    return small_sort(dtype, coords, n, k, k, o, s);
}

// The handle of a small cloud: perm0, the rank records (rec, k >= 2) or, with
// sel_keys, the key planes in array-0 order instead; m and the error bits.
// work: small_presort_words(n, k) words.
size_t small_presort_words(int n, int k) { return (size_t)2 * k * n; }
cudaError_t launch_small_presort(int dtype, const void* coords, int n, int k, uint32_t* work, const AllPlanes& rec,
                                 uint32_t* perm0, void* sel_keys, int64_t sel_stride, int64_t* m_out, int* err,
                                 cudaStream_t s) {
    SmallOut o{};
    o.arr_stride = o.inv_stride = n;
    o.m64 = m_out;
    o.err = err;
    const unsigned blocks = (unsigned)((n + 255) / 256);
    if (sel_keys) {
        o.arr = perm0;
        cudaError_t e = small_sort(dtype, coords, n, k, 1, o, s);
        if (e != cudaSuccess) return e;
        if (dtype == 0)
            k_small_keys<int32_t, uint32_t><<<blocks, 256, 0, s>>>(m_out, k, (const int32_t*)coords, perm0,
                                                                   (uint32_t*)sel_keys, sel_stride);
        else if (dtype == 1)
            k_small_keys<int64_t, uint64_t><<<blocks, 256, 0, s>>>(m_out, k, (const int64_t*)coords, perm0,
                                                                   (uint64_t*)sel_keys, sel_stride);
        else
            k_small_keys<float, uint32_t><<<blocks, 256, 0, s>>>(m_out, k, (const float*)coords, perm0,
                                                                 (uint32_t*)sel_keys, sel_stride);
        return cudaGetLastError();
    }
    o.arr = work;
    o.inv = work + (size_t)k * n;
    cudaError_t e = small_sort(dtype, coords, n, k, k, o, s);
    if (e != cudaSuccess) return e;
    k_small_recs<<<dim3(blocks, k), 256, 0, s>>>(m_out, k, o.arr, o.inv, n, rec, perm0);
    return cudaGetLastError();
}

template <typename T, typename KW, int NW, int E>
static cudaError_t init_small_as() {
    return cudaFuncSetAttribute((const void*)k_small_sort<T, KW, NW, E>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)small_smem<KW, NW, E>());
}
template <typename T, typename KW>
static cudaError_t init_small_of() {
    cudaError_t e = init_small_as<T, KW, 32, 4>();
    if (e == cudaSuccess) e = init_small_as<T, KW, 32, 8>();
    if (e == cudaSuccess) e = init_small_as<T, KW, 32, 16>();
    return e;
}
cudaError_t init_small_kernels() {
    cudaError_t e = init_small_of<int32_t, uint32_t>();
    if (e == cudaSuccess) e = init_small_of<int64_t, uint64_t>();
    if (e == cudaSuccess) e = init_small_of<float, uint32_t>();
    return e;
}

}  // namespace kd

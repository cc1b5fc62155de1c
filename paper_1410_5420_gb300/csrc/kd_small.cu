// kd_small.cu -- presort of a small cloud, one thread block per super key and
// chunk of tuples.
//
// Section 2.1's presort (k index arrays sorted by the cyclic super keys,
// duplicate tuples removed) for clouds of at most SMALL_MAX tuples, where a
// sort pass over the whole GPU is all launch latency:
//   k_small_sort     at most SMALL_ONE tuples: block d sorts the tuple
//                    indices by super key d in shared memory and removes
//                    duplicates;
//   k_small_chunks   more: block (c, d) sorts chunk c by super key d;
//   k_small_merge    every tuple's place among all chunks, by binary search
//                    in the others, and whether it is a duplicate;
//   k_small_compact  the places without the duplicates';
//   k_small_recs     the rank records the build reads, from the arrays and
//                    their inverses;
//   k_small_keys     the key planes in array-0 order (median-selection build).
// kd_presort_noalloc is all but the last two: 16384 float32 tuples of k = 3 in
// 29 us (in one block per super key 83; by a bitonic sort 284).
#include <cstdint>

#include "kd_block_sort.cuh"

namespace kd {

constexpr int SMALL_ONE = 2048;    // most tuples sorted by one block per super key
constexpr int SMALL_MAX = 196608;  // most tuples sorted in chunks
constexpr int SMALL_RUN = 32;      // longest run of equal x_d ordered by compares
// Runs that are not merged (small_runs): long ones of all but one super key
// from so many coordinates, ...
constexpr int64_t SMALL_LONG_RUNS = 350000;
// ... of half of them from so many tuples, and there all runs from so many
// coordinates.
constexpr int SMALL_MANY = 150000;
constexpr int64_t SMALL_RUNS = 1100000;
// Chunks of 2048 tuples up to 16384, 4096 up to 65536, 8192 above: a block's
// sort takes longer with its chunk, the merge with the number of chunks.
// Presorts of k = 3: 16384 float32 in chunks of 2048 52 us, of 4096 60; 30000
// int64 74 and 63; 40000 int64 in chunks of 4096 74, of 8192 87; 100000 float32
// 130 and 112.
__host__ __device__ constexpr int small_chunk(int n) { return n <= 16384 ? 2048 : (n <= 65536 ? 4096 : 8192); }

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

// Shared memory of one block's sort of at most 32 NW E tuples.
template <typename KW, int NW, int E>
struct SmallShared {
    uint32_t* key;   // the word being sorted ...
    KW* full;        // ... then x_d in its order (the same memory)
    uint16_t* idx;   // the order
    uint16_t (*wc)[RADIX];
    uint32_t *ws, *w;  // 32 and 4 words
};

template <typename T>
__device__ __forceinline__ bool small_nan(const T* __restrict__ coords, int count, int nt) {
    bool nan = false;
    if constexpr (sizeof(T) == 4 && T(0.5) != T(0))  // floats
        for (int i = threadIdx.x; i < count; i += nt) nan |= coords[i] != coords[i];
    return nan;
}

// The indices of n tuples (at most 32 NW E) by super key d.  First a stable
// radix sort by the leading differing bits of x_d (16, or 24 above 1024
// tuples: with 16, clustered floats leave runs too long for compares); then runs of equal words are ordered by the super key and the
// index by compares, or, where a run exceeds SMALL_RUN, everything is sorted
// again by the whole super key, least significant coordinate first, over
// the bytes that differ.  Bound by shared-memory latency and issue on its
// one SM.  Where a run exceeds SMALL_RUN, or most threads hold a tuple of a
// run, thread 0 calls report(whether it is the former), and stops what is left
// to do where that returns true.
template <typename T, typename KW, int NW, int E, typename R>
__device__ __forceinline__ void small_order(const T* __restrict__ coords, int n, int k, int d,
                                            const SmallShared<KW, NW, E>& S, const R& report) {
    constexpr int NT = 32 * NW, BITS = NT * E <= 1024 ? 16 : 24;
    uint32_t* const s_key = S.key;
    KW* const s_full = S.full;
    uint16_t* const s_idx = S.idx;
    uint16_t(*const wc)[RADIX] = S.wc;
    uint32_t *const s_ws = S.ws, *const s_w = S.w;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int base = warp * 32 * E + lane;  // place of row 0's element
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
            if (__syncthreads_or(threadIdx.x == 0 && report(true))) return;
            for (int r = k - 1; r >= 0; --r) {
                sort_by(d + r < k ? d + r : d + r - k, r == k - 1);
                __syncthreads();
            }
            fill_keys();
        } else if (const int ties = __syncthreads_count(tie)) {
            if (2 * ties > NT && threadIdx.x == 0) report(false);
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
}

// Whether tuples i and j are equal.
template <typename T>
__device__ __forceinline__ bool small_equal(const T* __restrict__ coords, int k, int i, int j) {
    for (int c = 0; c < k; ++c)
        if (small_key(coords[(int64_t)i * k + c]) != small_key(coords[(int64_t)j * k + c])) return false;
    return true;
}

#define SMALL_SHARED(KW, NW, E)                                                                                       \
    extern __shared__ __align__(16) unsigned char ssm[];                                                              \
    __shared__ __align__(16) uint16_t s_wc[NW][RADIX];                                                                \
    __shared__ uint32_t s_ws[32], s_w[4];                                                                             \
    uint16_t* const s_idx = reinterpret_cast<uint16_t*>(ssm + sizeof(KW) * 32 * NW * E);                              \
    KW* const s_full = reinterpret_cast<KW*>(ssm);                                                                    \
    const SmallShared<KW, NW, E> S{reinterpret_cast<uint32_t*>(ssm), s_full, s_idx, s_wc, s_ws, s_w}

// Block d: super key d's array of at most 32 NW E tuples, complete.
template <typename T, typename KW, int NW, int E>
__global__ void __launch_bounds__(32 * NW, 1) k_small_sort(const T* __restrict__ coords, int n, int k,
                                                           const SmallOut out) {
    constexpr int NT = 32 * NW;
    SMALL_SHARED(KW, NW, E);
    const int d = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int base = warp * 32 * E + lane;
    if (__syncthreads_or(small_nan(coords, n * k, NT))) {
        if (d == 0 && tid == 0) {
            if (out.err) atomicOr(out.err, ERR_NAN);
            if (out.m32) *out.m32 = -6;
        }
        return;
    }
    small_order(coords, n, k, d, S, [](bool) { return false; });
    // a tuple equal to its predecessor goes (the smallest index comes first)
    uint32_t keep[E], cnt = 0;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int o = base + e * 32;
        bool kp = o < n;
        if (kp && o > 0 && s_full[o - 1] == s_full[o]) {
            kp = !small_equal(coords, k, s_idx[o - 1], s_idx[o]);
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

// The super keys whose order in some chunk had runs (small_order): bit d a run
// of more than SMALL_RUN, bit 8 + d most tuples in runs.  Where `need` of the
// super keys under `mask` did, rows[1] is set and the merge, which tells equal
// x_d apart by the other coordinates at most steps of its searches, leaves the
// sort to the caller.  rows NULL: it takes any.
struct SmallRuns {
    int32_t* rows;
    uint32_t mask;
    int need;
};
__device__ __forceinline__ bool small_leave(const SmallRuns& R) { return R.rows && R.rows[1]; }

// Workspace of the chunked sort (rows of n per super key).
template <typename KW>
struct SmallWork {
    KW* key;         // x_d of every chunk's tuples in its order
    uint32_t* id;    // their indices
    uint32_t* raw;   // all indices in super-key-d order
    uint32_t* dup;   // bit per place of raw: a duplicate (rows of `words`)
    uint32_t* nan;   // per chunk: it holds a NaN
    int words;
    SmallRuns runs;
};

// Block (c, d): chunk c by super key d.
template <typename T, typename KW, int NW, int E>
__global__ void __launch_bounds__(32 * NW, 1) k_small_chunks(const T* __restrict__ coords, int n, int k,
                                                             const SmallWork<KW> W) {
    constexpr int CH = 32 * NW * E;
    SMALL_SHARED(KW, NW, E);
    const int c = blockIdx.x, d = blockIdx.y, tid = threadIdx.x;
    const int first = c * CH, cnt = min(n - first, CH);
    pdl_trigger();
    const T* x = coords + (int64_t)first * k;
    if (d == 0) {
        const int nan = __syncthreads_or(small_nan(x, cnt * k, CH / E));
        if (tid == 0) W.nan[c] = nan ? 1u : 0u;
    }
    for (int i = tid; i * 32 < cnt; i += CH / E) W.dup[(int64_t)d * W.words + first / 32 + i] = 0;
    small_order(x, cnt, k, d, S, [&](bool longer) {
        if (!W.runs.rows) return false;
        const uint32_t bit = 1u << (longer ? d : 8 + d);
        const uint32_t r = ((uint32_t)atomicOr(W.runs.rows, (int32_t)bit) | bit) & W.runs.mask;
        const bool enough = __popc((r | r >> 8) & 0xffu) >= W.runs.need;
        if (enough) W.runs.rows[1] = 1;
        return enough;  // no merge will follow
    });
    for (int i = tid; i < cnt; i += CH / E) {
        W.key[(int64_t)d * n + first + i] = s_full[i];
        W.id[(int64_t)d * n + first + i] = (uint32_t)(first + s_idx[i]);
    }
}

// Row d: the place in super-key-d order of the tuple at place q of the
// chunks' orders, and whether an equal tuple precedes it.  Equal x_d are
// told apart by the other coordinates and the index (that of an earlier
// chunk is smaller).
constexpr int SMALL_WAYS = 4;  // chunks searched side by side
// (Six blocks per SM: at five, of 48 registers, 65536 tuples of k = 3 over 16
// values took 378 us, 319 at six.)
template <typename T, typename KW>
__global__ void __launch_bounds__(256) k_small_merge(const T* __restrict__ coords, int n, int k, int chunk,
                                                     const SmallWork<KW> W) {
    const int q = blockIdx.x * 256 + threadIdx.x, d = blockIdx.y;
    pdl_wait();
    pdl_trigger();
    if (q >= n) return;
    const KW* key = W.key + (int64_t)d * n;
    const uint32_t* id = W.id + (int64_t)d * n;
    const KW x = key[q];
    const int me = (int)id[q], mc = q / chunk;
    // (no chunks rather than a return, whose extra registers cost a block per SM:
    // 196000 float32 tuples of k = 8 319 -> 380 us here)
    const int nc = small_leave(W.runs) ? 0 : (n + chunk - 1) / chunk;
    auto before = [&](int other) {  // equal x_d: the other tuple precedes this one
        for (int r = 1; r < k; ++r) {
            const int c = d + r < k ? d + r : d + r - k;
            const KW a = small_key(coords[(int64_t)other * k + c]), b = small_key(coords[(int64_t)me * k + c]);
            if (a != b) return a < b;
        }
        return other < me;
    };
    int rank = q - mc * chunk;
    bool dup = nc > 0 && rank > 0 && key[q - 1] == x && small_equal(coords, k, (int)id[q - 1], me);
    for (int c0 = 0; c0 < nc; c0 += SMALL_WAYS) {
        int pos[SMALL_WAYS], len[SMALL_WAYS];
#pragma unroll
        for (int u = 0; u < SMALL_WAYS; ++u) {
            const int c = c0 + u;
            pos[u] = 0;
            len[u] = c < nc && c != mc ? min(n - c * chunk, chunk) : 0;
        }
        for (int step = chunk; step > 0; step >>= 1) {
            KW y[SMALL_WAYS];
#pragma unroll
            for (int u = 0; u < SMALL_WAYS; ++u)
                y[u] = pos[u] + step <= len[u] ? key[(c0 + u) * chunk + pos[u] + step - 1] : (KW)0;
#pragma unroll
            for (int u = 0; u < SMALL_WAYS; ++u)
                if (pos[u] + step <= len[u] &&
                    (y[u] < x || (y[u] == x && before((int)id[(c0 + u) * chunk + pos[u] + step - 1]))))
                    pos[u] += step;
        }
#pragma unroll
        for (int u = 0; u < SMALL_WAYS; ++u) {
            rank += pos[u];
            const int p = (c0 + u) * chunk + pos[u] - 1;  // the last tuple before this one
            if (c0 + u < mc && pos[u] > 0 && key[p] == x) dup = dup || small_equal(coords, k, (int)id[p], me);
        }
    }
    W.raw[(int64_t)d * n + rank] = (uint32_t)me;
    if (dup) atomicOr(&W.dup[(int64_t)d * W.words + (rank >> 5)], 1u << (rank & 31));
}

// Row d: the kept tuples of 1024 places of raw to their places without the
// duplicates before them.
template <typename KW>
__global__ void __launch_bounds__(256) k_small_compact(int n, int nchunks, const SmallWork<KW> W, const SmallOut out) {
    __shared__ uint32_t s_sum[8], s_pre[32];
    const int d = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int p0 = blockIdx.x * 1024, w0 = p0 / 32;
    pdl_wait();
    pdl_trigger();
    if (small_leave(W.runs)) return;
    if (__syncthreads_or(tid < nchunks && W.nan[tid])) {
        if (d == 0 && blockIdx.x == 0 && tid == 0) {
            if (out.err) atomicOr(out.err, ERR_NAN);
            if (out.m32) *out.m32 = -6;
        }
        return;
    }
    const uint32_t* bits = W.dup + (int64_t)d * W.words;
    uint32_t v = 0;  // duplicates before p0
    for (int i = tid; i < w0; i += 256) v += __popc(bits[i]);
    v = __reduce_add_sync(0xffffffffu, v);
    if (lane == 0) s_sum[warp] = v;
    __syncthreads();
    if (warp == 0) {
        const uint32_t own = (w0 + lane) * 32 < n ? __popc(bits[w0 + lane]) : 0u;
        uint32_t x = own;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        const uint32_t pre = __reduce_add_sync(0xffffffffu, lane < 8 ? s_sum[lane] : 0u);
        s_pre[lane] = pre + x - own;
        if (lane == 31 && d == 0 && p0 + 1024 >= n) {
            const uint32_t m = (uint32_t)n - (pre + x);
            if (out.m64) *out.m64 = m;
            if (out.m32) *out.m32 = (int32_t)m;
        }
    }
    __syncthreads();
    for (int r = 0; r < 4; ++r) {
        const int w = r * 8 + warp, p = p0 + w * 32 + lane;
        if (p >= n) break;
        const uint32_t b = bits[w0 + w];
        if ((b >> lane) & 1u) continue;
        const uint32_t o = (uint32_t)p - (s_pre[w] + __popc(b & lanemask_lt()));
        const uint32_t t = W.raw[(int64_t)d * n + p];
        out.arr[d * out.arr_stride + o] = t;
        if (out.inv) out.inv[d * out.inv_stride + t] = o;
    }
}

// rec[d][p][i] = place in array p of the tuple at place i of array d (p != d;
// array 0 also its own places), and perm0 = array 0.  Block row y: array d.
__global__ void __launch_bounds__(256) k_small_recs(const int64_t* __restrict__ m_ptr, int k,
                                                    const uint32_t* __restrict__ arr, const uint32_t* __restrict__ inv,
                                                    int64_t stride, const __grid_constant__ AllPlanes rec,
                                                    uint32_t* __restrict__ perm0) {
    const int i = blockIdx.x * 256 + threadIdx.x, d = blockIdx.y;
    pdl_wait();
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

// Words of the chunked sort's workspace for narrays super keys.
static int64_t small_rows(int64_t n, int narrays) { return (int64_t)narrays * ((n + 3) & ~(int64_t)3); }
static int small_dup_words(int n) { return (n + 31) / 32; }
static size_t small_work_words(int dtype, int n, int narrays) {
    const size_t rows = (size_t)small_rows(n, narrays);
    return rows * ((dtype == 1 ? 2 : 1) + 2) + (size_t)narrays * small_dup_words(n) + 32;
}

template <typename T, typename KW, int NW, int E>
static cudaError_t small_sort_as(const void* coords, int n, int k, int narrays, const SmallOut& out, cudaStream_t s) {
    // (the error of the launch call itself: one pending from earlier work is neither reported nor cleared)
    const T* c = static_cast<const T*>(coords);
    SmallOut o = out;
    void* argv[] = {&c, &n, &k, &o};
    return cudaLaunchKernel(reinterpret_cast<const void*>(&k_small_sort<T, KW, NW, E>), dim3(narrays), dim3(32 * NW),
                            argv, small_smem<KW, NW, E>(), s);
}

template <typename T, typename KW, int NW, int E>
static cudaError_t small_chunks_as(const void* coords, int n, int k, int narrays, const SmallWork<KW>& W,
                                   cudaStream_t s) {
    const T* c = static_cast<const T*>(coords);
    SmallWork<KW> w = W;
    void* argv[] = {&c, &n, &k, &w};
    const int ch = 32 * NW * E;
    return cudaLaunchKernel(reinterpret_cast<const void*>(&k_small_chunks<T, KW, NW, E>),
                            dim3((n + ch - 1) / ch, narrays), dim3(32 * NW), argv, small_smem<KW, NW, E>(), s);
}

// One block per super key up to SMALL_ONE tuples, of 8 warps up to 1024 (its
// barriers and scans are shorter); chunks above (work: small_work_words).
template <typename T, typename KW>
static cudaError_t small_sort_of(const void* coords, int n, int k, int narrays, uint32_t* work, const SmallOut& out,
                                 const SmallRuns& runs, cudaStream_t s) {
    if (n <= 256) return small_sort_as<T, KW, 8, 1>(coords, n, k, narrays, out, s);
    if (n <= 1024) return small_sort_as<T, KW, 8, 4>(coords, n, k, narrays, out, s);
    if (n <= SMALL_ONE) return small_sort_as<T, KW, 32, 2>(coords, n, k, narrays, out, s);
    const int64_t rows = small_rows(n, narrays);
    SmallWork<KW> W;
    W.key = reinterpret_cast<KW*>(work);
    W.id = work + rows * (sizeof(KW) / 4);
    W.raw = W.id + rows;
    W.dup = W.raw + rows;
    W.words = small_dup_words(n);
    W.nan = W.dup + (int64_t)narrays * W.words;
    W.runs = runs;
    const int chunk = small_chunk(n);
    cudaError_t e = chunk == 2048 ? small_chunks_as<T, KW, 32, 2>(coords, n, k, narrays, W, s)
                    : chunk == 4096 ? small_chunks_as<T, KW, 32, 4>(coords, n, k, narrays, W, s)
                                    : small_chunks_as<T, KW, 32, 8>(coords, n, k, narrays, W, s);
    if (e == cudaSuccess)
        e = launch_dependent(k_small_merge<T, KW>, dim3((n + 255) / 256, narrays), dim3(256), 0, s, (const T*)coords, n,
                             k, chunk, W);
    if (e == cudaSuccess)
        e = launch_dependent(k_small_compact<KW>, dim3((n + 1023) / 1024, narrays), dim3(256), 0, s, n,
                             (n + chunk - 1) / chunk, W, out);
    return e;
}

static cudaError_t small_sort(int dtype, const void* coords, int n, int k, int narrays, uint32_t* work,
                              const SmallOut& out, const SmallRuns& runs, cudaStream_t s) {
    if (n < 1 || n > SMALL_MAX) return cudaErrorInvalidValue;
    if (dtype == 0) return small_sort_of<int32_t, uint32_t>(coords, n, k, narrays, work, out, runs, s);
    if (dtype == 1) return small_sort_of<int64_t, uint64_t>(coords, n, k, narrays, work, out, runs, s);
    return small_sort_of<float, uint32_t>(coords, n, k, narrays, work, out, runs, s);
}

// Kernels launched by one sort.
int small_sort_launches(int64_t n) { return n <= SMALL_ONE ? 1 : 3; }
// Whether the sort reads the coordinates while it writes its outputs.
bool small_reads_while_writing(int64_t n) { return n <= SMALL_ONE; }

// kd_presort_noalloc: rows of n in out, m (or KD_ENAN) in m_out; work:
// small_arrays_bytes(n, k) bytes.
size_t small_arrays_bytes(int n, int k) { return n <= SMALL_ONE ? 0 : small_work_words(1, n, k) * 4; }
cudaError_t launch_small_arrays(int dtype, const void* coords, int n, int k, void* work, int32_t* rows, int32_t* m_out,
                                cudaStream_t s) {
    SmallOut o{};
    o.arr = reinterpret_cast<uint32_t*>(rows);
    o.arr_stride = n;
    o.m32 = m_out;
    return small_sort(dtype, coords, n, k, k, static_cast<uint32_t*>(work), o, SmallRuns{}, s);
}

// Which runs send a whole presort (all k arrays) back to the caller: the work
// of the merge grows with the tuples, the chunks and the dimensions, that of
// the digit passes hardly, and constant bytes save them passes.  Whole builds,
// by digit passes and merged: 65536 int64 tuples of k = 8 over 2 values per
// coordinate 0.63 and 1.72 ms (16 values 0.66 and 0.88, 64 values 0.65 and 0.71),
// 196000 of k = 3 over 64 values 0.45 and 0.83, of k = 8 over 2 values 0.90 and
// 6.89; 40000 of k = 8 over 16 values 0.66 and 0.58.  With three values in half
// of the coordinates: 196000 of k = 6 0.75 and 1.45, 100000 float32 of k = 8 0.99
// and 0.94.  Over 1000 values (short runs): 196000 int64 of k = 8 1.00 and 1.53,
// 140000 float32 of k = 8 1.14 and 0.95.  What is left has cost its block sorts
// and a read back, 0.06 to 0.1 ms.
static SmallRuns small_runs(int n, int k, int32_t* rows) {
    const int64_t nk = (int64_t)n * k;
    const bool many = n > SMALL_MANY;
    SmallRuns r{};
    r.mask = k < 3 ? 0u : (nk > SMALL_LONG_RUNS ? 0xffu : 0u) | (many && nk > SMALL_RUNS ? 0xff00u : 0u);
    r.need = many ? (k + 1) / 2 : k - 1;
    r.rows = r.mask ? rows : nullptr;
    return r;
}
// The handle of a small cloud: perm0, the rank records (rec, k >= 2) or, with
// sel_keys, the key planes in array-0 order instead; m and the error bits.
// work: small_presort_words words (the sort's, then the arrays and their
// inverses).
size_t small_presort_words(int dtype, int n, int k, bool all_arrays) {
    return (n <= SMALL_ONE ? 0 : (small_work_words(dtype, n, all_arrays ? k : 1) + 3) / 4 * 4) +
           (all_arrays ? (size_t)2 * k * n : 0);
}
cudaError_t launch_small_presort(int dtype, const void* coords, int n, int k, uint32_t* work, const AllPlanes& rec,
                                 uint32_t* perm0, void* sel_keys, int64_t sel_stride, int64_t* m_out, int32_t* runs,
                                 int* err, cudaStream_t s) {
    SmallOut o{};
    o.arr_stride = o.inv_stride = n;
    o.m64 = m_out;
    o.err = err;
    const unsigned blocks = (unsigned)((n + 255) / 256);
    if (sel_keys) {
        o.arr = perm0;
        cudaError_t e = small_sort(dtype, coords, n, k, 1, work, o, SmallRuns{}, s);
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
    o.arr = work + small_presort_words(dtype, n, k, true) - (size_t)2 * k * n;
    o.inv = o.arr + (size_t)k * n;
    cudaError_t e = small_sort(dtype, coords, n, k, k, work, o, small_runs(n, k, runs), s);
    if (e != cudaSuccess) return e;
    return launch_dependent(k_small_recs, dim3(blocks, k), dim3(256), 0, s, (const int64_t*)m_out, k,
                            (const uint32_t*)o.arr, (const uint32_t*)o.inv, (int64_t)n, rec, perm0);
}

template <typename T, typename KW>
static cudaError_t init_small_of() {
    cudaError_t e = cudaFuncSetAttribute((const void*)k_small_chunks<T, KW, 32, 4>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)small_smem<KW, 32, 4>());
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute((const void*)k_small_chunks<T, KW, 32, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)small_smem<KW, 32, 8>());
    return e;
}
cudaError_t init_small_kernels() {
    cudaError_t e = init_small_of<int32_t, uint32_t>();
    if (e == cudaSuccess) e = init_small_of<int64_t, uint64_t>();
    if (e == cudaSuccess) e = init_small_of<float, uint32_t>();
    return e;
}

}  // namespace kd

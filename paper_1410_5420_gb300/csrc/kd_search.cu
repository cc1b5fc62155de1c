// kd_search.cu -- searches over a built tree: m nearest neighbours and
// region search (the "Nearest Neighbors" subsection and the region search
// of the source-code subsection of the paper).
//
// A search index holds the tree's tuples in address order (one plane per
// coordinate, so that 32 lanes reading 32 consecutive addresses coalesce)
// and the tuple index of every node.  The tree is the
// in-order layout the builder writes: the subtree of a node covers a
// contiguous address range [lo, hi], its node is the median lo + (hi-lo)/2,
// its children cover [lo, mid-1] and [mid+1, hi], and the split dimension
// of depth t is t mod k.  A subtree on the "less" side holds only tuples
// with x_d <= the node's x_d, the "greater" side only x_d >= (super keys
// order ties by the next coordinates), which is what both searches prune on.
//
//   k_index_gather  planes of the tuples' coordinates in address order
//   k_boxes         bounding boxes over blocks of 32 consecutive addresses
//   k_knn           one warp per query: walk of the box tree, nearest first,
//                   the best candidates sorted across the warp
//   k_knn_exact     the queries k_knn has left (distances that 32-bit floats
//                   do not tell apart), by double distances alone
//   k_knn_walk      one thread per query: depth-first walk of the tree, for
//                   an index without boxes
//   k_region        one thread per box: depth-first walk visiting a side
//                   only if the box reaches it; counts, then (second launch
//                   after a scan of the counts) the indices
//
// Distances are defined exactly (no fused multiply-add): per dimension the
// absolute difference (integers: |a - b| as an unsigned 64-bit value,
// rounded to double; floats: the double difference of the two values),
// squared and summed in double in dimension order.
#include <algorithm>
#include <memory>
#include <mutex>
#include <string>
#include <type_traits>
#include <vector>

#include "kd_internal.cuh"
#include "kdtree.h"

namespace kd {
int ctx_device(const kd_ctx* ctx);
cudaStream_t ctx_stream(const kd_ctx* ctx);
void ctx_set_error(kd_ctx* ctx, const std::string& msg);
void ctx_add_launches(kd_ctx* ctx, int n);
kd_status ctx_alloc(kd_ctx* ctx, void** p, size_t bytes);
void ctx_free(kd_ctx* ctx, void* p);
std::recursive_mutex& ctx_mutex(kd_ctx* ctx);
}  // namespace kd

struct kd_index_s {
    kd_ctx* ctx = nullptr;
    int64_t m = 0;
    int k = 0;
    int dtype = 0;
    void* pts = nullptr;  // k planes of m words, address order, input dtype
    int32_t* node_tuple = nullptr;
    void* boxes = nullptr;  // bounding boxes of every level (nullptr: they did not fit the budget)
    int64_t box_off[5] = {};  // level l: first word in boxes ...
    int32_t nbox[5] = {};     // ... and number of boxes
    int top = 0;
    bool dense = false;  // integers that fill a good part of their range (index_dense)
};

namespace {

using kd::ERR_INTERNAL;
using kd::ERR_NAN;
using kd::MAXK;

constexpr int SEARCH_THREADS = 128;
constexpr int STACK_MAX = 64;  // a tree of at most 2^30 nodes is at most 31 levels deep
constexpr int REGION_KEEP = 16;   // tuples of a box kept by the counting walk
constexpr int REGION_STACK = 32;  // at most one waiting side per level

template <typename T>
__device__ __forceinline__ double abs_diff(T a, T b);
template <>
__device__ __forceinline__ double abs_diff<int32_t>(int32_t a, int32_t b) {
    const int64_t x = a, y = b;
    return __ull2double_rn(x > y ? (uint64_t)(x - y) : (uint64_t)(y - x));
}
template <>
__device__ __forceinline__ double abs_diff<int64_t>(int64_t a, int64_t b) {
    return __ull2double_rn(a > b ? (uint64_t)a - (uint64_t)b : (uint64_t)b - (uint64_t)a);
}
template <>
__device__ __forceinline__ double abs_diff<float>(float a, float b) {
    return fabs(__dsub_rn((double)a, (double)b));
}

template <typename T>
__device__ __forceinline__ bool is_nan(T) { return false; }
template <>
__device__ __forceinline__ bool is_nan<float>(float v) { return v != v; }

// pts[d * m + a] = coordinate d of the tuple at address a.
template <typename T>
__global__ void __launch_bounds__(256) k_index_gather(const T* __restrict__ coords, const int32_t* __restrict__ tuple,
                                                      int64_t m, int k, int64_t n, T* __restrict__ pts,
                                                      int* __restrict__ err) {
    for (int64_t a = (int64_t)blockIdx.x * 256 + threadIdx.x; a < m; a += (int64_t)gridDim.x * 256) {
        const int32_t t = tuple[a];
        if (t < 0 || t >= n) {
            atomicOr(err, ERR_INTERNAL);
            continue;
        }
        for (int d = 0; d < k; ++d) pts[d * m + a] = coords[(int64_t)t * k + d];
    }
}

// ---------------------------------------------------- nearest neighbours
// Address order is spatially coherent (it is the tree's in-order), so every
// 32 consecutive tuples are a compact block.  Over these blocks lies a tree
// of bounding boxes with 32 children per node: level 0 holds the boxes of
// the blocks, level l + 1 one box per 32 boxes of level l.  One warp answers
// one query: at a node every lane tests one child's box, the children are
// entered nearest first, and in a block every lane computes one distance.
// The best candidates so far lie sorted across the warp, one per lane
// (KD_KNN_MAX = 32 of them).
//
// What bounded the one-thread-per-query walk this replaces: at two FP64
// lanes per cycle and SM the double distance of every visited tuple, the
// neighbour list and the stack in local memory, and, for clustered points, a
// few queries whose split-plane bounds let them walk most of a dense cluster
// while the rest of the GPU had finished.  Here candidates are kept by a
// float distance and only the at most 32 survivors get the double one; the
// boxes bound by the distance to the tuples themselves.  Eight neighbours of
// each of 2^22 int64 tuples: 33.9 -> 7.05 ms, now bound by instruction issue
// (5.7 blocks, 4.7 nodes and 1.1 sorts per query); five of 100003 float32
// queries among 10^6 clustered tuples: 3.5-28 ms (by the cluster geometry)
// -> 0.6.
//
// Float distances.  a = the float sum of the squared float |p - q| differs
// from the exact distance t by less than 2^-20 t (roundings of at most
// (K + 4) 2^-24 in all), unless it underflows (below KNN_TINY) or overflows to
// +inf.  So with A the kn-th smallest a, every one of the kn nearest tuples has
// a <= A (1 + 2^-18) = the bound, and a box whose float distance, less
// 2^-18 of itself, exceeds the bound holds none of them.  All candidates up
// to the bound are ranked by (double distance, tuple index).  If more than
// the list's 32 lie below it (ties, or near ties, around kn), the query is
// answered again with double distances for every candidate (EXACT).  Where
// that is certain because the bound cannot fall any more (KNN_TINY) or tells
// nothing apart (+inf), the walk gives up and leaves the query to
// k_knn_exact, which prunes by double distances of the boxes too: each of
// their rounded steps grows with its operands, so that no tuple of a box comes
// out nearer than the box.  2^17 normal float32 tuples scaled by 1e-20 or by
// 1e22, whose squares leave the float's range, eight neighbours of each: 3.0
// ms (both float walks over every block of the index 754 ms, the walk by one
// thread per query 8.0, unscaled 0.23).
constexpr int BOX_W = 32;        // tuples per block, children per node
constexpr int BOX_LEVELS = 5;    // level 4 has at most 32 boxes for 2^30 tuples
constexpr int KNN_THREADS = 256;
constexpr float KNN_MARGIN = 3.814697265625e-6f;  // 2^-18
constexpr float KNN_TINY = 1e-35f;
constexpr uint32_t KNN_NONE = 0xffffffffu;  // no candidate / child done
constexpr uint32_t KNN_OPEN = 0xfffffffeu;  // bound while the list holds fewer than kn
constexpr uint32_t KNN_INF = 0x7f800000u;   // float bits of +inf
constexpr int32_t KNN_LEFT = INT32_MIN;     // first index of a row that is left to k_knn_exact

template <typename T>
struct KnnTree {
    const T* pts;  // k planes of `stride` words, address order
    int64_t stride;
    const int32_t* tuple;
    int32_t m;
    int k;
    int top;  // the level whose boxes (at most 32) are tested first
    // boxes of level l, 32 siblings side by side: word (g * 2k + d) * 32 + c
    // is the lower bound in dimension d of child c of node g, d + k the upper
    const T* box[BOX_LEVELS];
    int32_t nbox[BOX_LEVELS];
};

// An unsigned difference as a float, within 2^-23 of it.  (64 bits: from the
// two halves, three roundings; the conversion instruction for 64-bit
// integers runs on the FP64 pipe, which it kept 92% busy.)
__device__ __forceinline__ float udiff_f(uint32_t u) { return __uint2float_rn(u); }
__device__ __forceinline__ float udiff_f(uint64_t u) {
    return fmaf(__uint2float_rn((uint32_t)(u >> 32)), 4294967296.0f, __uint2float_rn((uint32_t)u));
}
// |a - b| as such a float (the float difference for floats).
template <typename T>
__device__ __forceinline__ float diff_f(T a, T b) {
    using U = typename std::make_unsigned<T>::type;
    return udiff_f(a > b ? (U)((U)a - (U)b) : (U)((U)b - (U)a));
}
template <>
__device__ __forceinline__ float diff_f<float>(float a, float b) { return __fsub_rn(a, b); }

// Distance of q from the interval [lo, hi], as diff_f.
template <typename T>
__device__ __forceinline__ float gap_f(T q, T lo, T hi) {
    using U = typename std::make_unsigned<T>::type;
    const U below = (U)lo - (U)q, above = (U)q - (U)hi;
    return udiff_f(q < lo ? below : (q > hi ? above : (U)0));
}
template <>
__device__ __forceinline__ float gap_f<float>(float q, float lo, float hi) {
    return q < lo ? __fsub_rn(lo, q) : (q > hi ? __fsub_rn(q, hi) : 0.0f);
}

__device__ __forceinline__ uint32_t knn_bound(float a) {
    return __float_as_uint(fmaxf(a * (1.0f + KNN_MARGIN), KNN_TINY));
}
// More candidates up to the bound than the list holds, and a bound that
// cannot fall any more or that tells nothing apart.  Asked once per 32 blocks
// of floats, once per 1024 of 64-bit integers (whose differences overflow only
// to the far ends of the type), never of 32-bit ones.  (In knn_block, or with a
// bound that also says so, k_knn has more spills and all neighbours of 2^22
// int64 tuples take 7.09 -> 7.33 to 7.49 ms; once per 32 blocks 7.16 -> 7.21.)
template <typename T>
constexpr bool knn_may_stick(int level) {
    return std::is_same<T, float>::value || (sizeof(T) == 8 && level > 1);
}
__device__ __forceinline__ bool knn_stuck(uint32_t lost, uint32_t bound) {
    return lost <= bound && (bound <= __float_as_uint(KNN_TINY) || bound >= KNN_INF);
}

// The query of one warp and its candidates (lane j: the j-th best).
template <typename T, int K>  // K: the dimensions, or MAXK: at most that many
struct KnnQuery {
    T q[K];
    int32_t self;    // address excluded, or -1
    int kn;
    uint32_t bound;  // float bits: nothing above it can be among the kn nearest
    uint32_t key;    // candidate: float bits of its distance ...
    int32_t addr;    // ... and address
    uint32_t lost;   // smallest float distance that did not fit the list
    uint64_t dkey;   // exact form: the double distance's bits and the tuple index
    int32_t tup;
};

template <typename T, int K>
__device__ __forceinline__ double exact_dist(const KnnTree<T>& X, const T (&q)[K], int32_t a) {
    double acc = 0.0;
#pragma unroll
    for (int d = 0; d < K; ++d) {
        if (K == MAXK && d >= X.k) break;
        const double u = abs_diff<T>(X.pts[d * X.stride + a], q[d]);
        acc = __dadd_rn(acc, __dmul_rn(u, u));
    }
    return acc;
}

// Ascending by key across the warp (bitonic).
__device__ __forceinline__ void warp_sort(uint32_t& key, int32_t& val) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int size = 2; size <= 32; size <<= 1) {
#pragma unroll
        for (int st = size >> 1; st > 0; st >>= 1) {
            const uint32_t ok = __shfl_xor_sync(0xffffffffu, key, st);
            const int32_t ov = __shfl_xor_sync(0xffffffffu, val, st);
            const bool up = ((lane & size) == 0) == ((lane & st) == 0);  // this lane keeps the smaller
            if (up ? ok < key : ok > key) {
                key = ok;
                val = ov;
            }
        }
    }
}

template <typename T, int K, bool EXACT>
__device__ __forceinline__ void knn_block(const KnnTree<T>& X, KnnQuery<T, K>& Q, int32_t blk) {
    const int lane = threadIdx.x & 31;
    const int32_t a = blk * BOX_W + lane;
    const bool ok = a < X.m && a != Q.self;
    float s = 0.0f;
    if (ok) {
#pragma unroll
        for (int d = 0; d < K; ++d) {
            if (K == MAXK && d >= X.k) break;
            const float u = diff_f(X.pts[d * X.stride + a], Q.q[d]);
            s = fmaf(u, u, s);
        }
    }
    const uint32_t key = __float_as_uint(s);
    const bool pass = ok && s == s && key <= Q.bound;  // (an infinite coordinate may give no distance: NaN)
    uint32_t mask = __ballot_sync(0xffffffffu, pass);
    if (mask == 0) return;
    if constexpr (EXACT) {
        uint64_t dk = 0;
        int32_t tp = 0;
        if (pass) {
            dk = (uint64_t)__double_as_longlong(exact_dist<T, K>(X, Q.q, a));
            tp = X.tuple[a];
        }
        for (; mask; mask &= mask - 1) {
            const int src = __ffs(mask) - 1;
            const uint64_t d = __shfl_sync(0xffffffffu, dk, src);
            const int32_t t = __shfl_sync(0xffffffffu, tp, src);
            const bool before = Q.dkey < d || (Q.dkey == d && Q.tup < t);
            const int pos = __popc(__ballot_sync(0xffffffffu, before));
            const uint64_t ud = __shfl_up_sync(0xffffffffu, Q.dkey, 1);
            const int32_t ut = __shfl_up_sync(0xffffffffu, Q.tup, 1);
            if (lane > pos) {
                Q.dkey = ud;
                Q.tup = ut;
            } else if (lane == pos) {
                Q.dkey = d;
                Q.tup = t;
            }
        }
        const uint64_t A = __shfl_sync(0xffffffffu, Q.dkey, Q.kn - 1);
        if (A != ~0ull) Q.bound = knn_bound(__double2float_ru(__longlong_as_double((long long)A)));
    } else {
        if (__popc(mask) > 8) {
            // many: sort them, then merge with the list (both ascending)
            uint32_t nk = pass ? key : KNN_NONE;
            int32_t na = a;
            warp_sort(nk, na);
            if (Q.bound == KNN_OPEN && __shfl_sync(0xffffffffu, Q.key, 0) == KNN_NONE) {  // the list is empty
                Q.key = nk;
                Q.addr = na;
                const uint32_t A0 = __shfl_sync(0xffffffffu, Q.key, Q.kn - 1);
                if (A0 != KNN_NONE) Q.bound = knn_bound(__uint_as_float(A0));
                return;
            }
            nk = __shfl_xor_sync(0xffffffffu, nk, 31);
            na = __shfl_xor_sync(0xffffffffu, na, 31);
            const bool take = nk < Q.key;
            const uint32_t out = take ? Q.key : nk;
            if (take) {
                Q.key = nk;
                Q.addr = na;
            }
            Q.lost = min(Q.lost, __reduce_min_sync(0xffffffffu, out));
#pragma unroll
            for (int st = 16; st > 0; st >>= 1) {
                const uint32_t ok2 = __shfl_xor_sync(0xffffffffu, Q.key, st);
                const int32_t oa = __shfl_xor_sync(0xffffffffu, Q.addr, st);
                if ((lane & st) == 0 ? ok2 < Q.key : ok2 > Q.key) {
                    Q.key = ok2;
                    Q.addr = oa;
                }
            }
        } else {
            for (; mask; mask &= mask - 1) {
                const int src = __ffs(mask) - 1;
                const uint32_t d = __shfl_sync(0xffffffffu, key, src);
                const int pos = __popc(__ballot_sync(0xffffffffu, Q.key <= d));
                const uint32_t uk = __shfl_up_sync(0xffffffffu, Q.key, 1);
                const int32_t ua = __shfl_up_sync(0xffffffffu, Q.addr, 1);
                Q.lost = min(Q.lost, pos == 32 ? d : __shfl_sync(0xffffffffu, Q.key, 31));
                if (lane > pos) {
                    Q.key = uk;
                    Q.addr = ua;
                } else if (lane == pos) {
                    Q.key = d;
                    Q.addr = blk * BOX_W + src;
                }
            }
        }
        const uint32_t A = __shfl_sync(0xffffffffu, Q.key, Q.kn - 1);
        if (A != KNN_NONE) Q.bound = knn_bound(__uint_as_float(A));
    }
}

// The children (boxes of level L) of node `node`, nearest first.
template <typename T, int K, bool EXACT, int L>
__device__ __forceinline__ void knn_node(const KnnTree<T>& X, KnnQuery<T, K>& Q, int32_t node) {
    if constexpr (L > 0) {
        if (L > X.top) {
            knn_node<T, K, EXACT, L - 1>(X, Q, 0);
            return;
        }
    }
    const int lane = threadIdx.x & 31;
    uint32_t key = KNN_NONE;
    if (node * BOX_W + lane < X.nbox[L]) {
        const T* b = X.box[L] + (int64_t)node * (2 * (K == MAXK ? X.k : K) * BOX_W) + lane;
        float s = 0.0f;
#pragma unroll
        for (int d = 0; d < K; ++d) {
            if (K == MAXK && d >= X.k) break;
            const float u = gap_f<T>(Q.q[d], b[d * BOX_W], b[((K == MAXK ? X.k : K) + d) * BOX_W]);
            s = fmaf(u, u, s);
        }
        key = __float_as_uint(s * (1.0f - KNN_MARGIN));
    }
    for (int i = 0; i < BOX_W; ++i) {
        const uint32_t best = __reduce_min_sync(0xffffffffu, key);
        if (best > Q.bound) break;
        const int c = __ffs(__ballot_sync(0xffffffffu, key == best)) - 1;
        if (lane == c) key = KNN_NONE;
        if constexpr (L > 0) {
            knn_node<T, K, EXACT, L - 1>(X, Q, node * BOX_W + c);
            if constexpr (!EXACT && knn_may_stick<T>(L))
                if (knn_stuck(Q.lost, Q.bound)) break;
        } else {
            knn_block<T, K, EXACT>(X, Q, node * BOX_W + c);
        }
    }
}

// ---- by double distances alone: one query, its list (distance bits, tuple
// index) sorted across the warp.
template <typename T, int K>
struct KnnExact {
    T q[K];
    int32_t self;
    int kn;
    uint64_t last;  // distance of the kn-th best (~0: fewer so far)
    uint64_t dkey;
    int32_t tup;
};

__device__ __forceinline__ uint64_t warp_min64(uint64_t x) {
    const uint32_t hi = __reduce_min_sync(0xffffffffu, (uint32_t)(x >> 32));
    const uint32_t lo = __reduce_min_sync(0xffffffffu, (uint32_t)(x >> 32) == hi ? (uint32_t)x : 0xffffffffu);
    return (uint64_t)hi << 32 | lo;
}

template <typename T, int K>
__device__ __forceinline__ void knn_exact_block(const KnnTree<T>& X, KnnExact<T, K>& Q, int32_t blk) {
    const int lane = threadIdx.x & 31;
    const int32_t a = blk * BOX_W + lane;
    double dist = 0.0;
    int32_t tp = 0;
    bool pass = a < X.m && a != Q.self;
    if (pass) {
        dist = exact_dist<T, K>(X, Q.q, a);
        tp = X.tuple[a];
    }
    const uint64_t dk = (uint64_t)__double_as_longlong(dist);
    pass = pass && dist == dist && dk <= Q.last;
    for (uint32_t mask = __ballot_sync(0xffffffffu, pass); mask; mask &= mask - 1) {
        const int src = __ffs(mask) - 1;
        const uint64_t d = __shfl_sync(0xffffffffu, dk, src);
        const int32_t t = __shfl_sync(0xffffffffu, tp, src);
        const int pos = __popc(__ballot_sync(0xffffffffu, Q.dkey < d || (Q.dkey == d && Q.tup < t)));
        if (pos >= Q.kn) continue;
        const uint64_t ud = __shfl_up_sync(0xffffffffu, Q.dkey, 1);
        const int32_t ut = __shfl_up_sync(0xffffffffu, Q.tup, 1);
        if (lane > pos) {
            Q.dkey = ud;
            Q.tup = ut;
        } else if (lane == pos) {
            Q.dkey = d;
            Q.tup = t;
        }
    }
    Q.last = __shfl_sync(0xffffffffu, Q.dkey, Q.kn - 1);
}

template <typename T, int K, int L>
__device__ __forceinline__ void knn_exact_node(const KnnTree<T>& X, KnnExact<T, K>& Q, int32_t node) {
    if constexpr (L > 0) {
        if (L > X.top) {
            knn_exact_node<T, K, L - 1>(X, Q, 0);
            return;
        }
    }
    const int lane = threadIdx.x & 31;
    uint64_t key = ~0ull;
    if (node * BOX_W + lane < X.nbox[L]) {
        const T* b = X.box[L] + (int64_t)node * (2 * (K == MAXK ? X.k : K) * BOX_W) + lane;
        double acc = 0.0;
#pragma unroll
        for (int d = 0; d < K; ++d) {
            if (K == MAXK && d >= X.k) break;
            const T lo = b[d * BOX_W], hi = b[((K == MAXK ? X.k : K) + d) * BOX_W];
            const double u = Q.q[d] < lo ? abs_diff<T>(lo, Q.q[d]) : (Q.q[d] > hi ? abs_diff<T>(Q.q[d], hi) : 0.0);
            acc = __dadd_rn(acc, __dmul_rn(u, u));
        }
        key = (uint64_t)__double_as_longlong(acc);
    }
    for (int i = 0; i < BOX_W; ++i) {
        const uint64_t best = warp_min64(key);
        if (best == ~0ull || best > Q.last) break;
        const int c = __ffs(__ballot_sync(0xffffffffu, key == best)) - 1;
        if (lane == c) key = ~0ull;
        if constexpr (L > 0) knn_exact_node<T, K, L - 1>(X, Q, node * BOX_W + c);
        else knn_exact_block<T, K>(X, Q, node * BOX_W + c);
    }
}

// The candidates of this lane's group of `width` lanes (address c of query
// qc, or c = -1) by (double distance, tuple index): the first kn to row qi.
template <typename T, int K>
__device__ __forceinline__ void knn_emit(const KnnTree<T>& X, const T* __restrict__ queries, int64_t qi, int32_t c,
                                         int width, int kn, int32_t* __restrict__ idx_out,
                                         double* __restrict__ d_out) {
    const int lane = threadIdx.x & 31, first = lane & ~(width - 1);
    uint64_t dk = ~0ull;
    int32_t tp = INT32_MAX;
    if (c >= 0) {
        T q[K];
#pragma unroll
        for (int d = 0; d < K; ++d) {
            if (K == MAXK && d >= X.k) break;
            q[d] = queries ? queries[qi * (K == MAXK ? X.k : K) + d] : X.pts[d * X.stride + qi];
        }
        dk = (uint64_t)__double_as_longlong(exact_dist<T, K>(X, q, c));
        tp = X.tuple[c];
    }
    int rank = 0;
    for (int j = 0; j < width; ++j) {
        const uint64_t d = __shfl_sync(0xffffffffu, dk, first + j);
        const int32_t t = __shfl_sync(0xffffffffu, tp, first + j);
        rank += (d < dk || (d == dk && t < tp)) ? 1 : 0;
    }
    const uint32_t group = width == 32 ? 0xffffffffu : ((1u << width) - 1u) << first;
    const int cnt = __popc(__ballot_sync(0xffffffffu, c >= 0) & group);
    if (c >= 0 ? rank < kn : (cnt > 0 && lane - first >= cnt && lane - first < kn)) {
        const int j = c >= 0 ? rank : lane - first;  // (rows past the last candidate: no tuple)
        idx_out[qi * kn + j] = c >= 0 ? tp : -1;
        if (d_out) d_out[qi * kn + j] = __longlong_as_double(c >= 0 ? (long long)dk : 0x7ff0000000000000ll);
    }
}

// queries == nullptr: every address is a query (row = its address) and its
// own tuple is not a candidate.  A warp answers 32 / width queries in turn
// (width: a power of two, at least kn) and then computes the double
// distances of all their candidates at once, one per lane: with kn = 8 and
// one query at a time, 24 of the 32 lanes of every FP64 instruction idled
// while that pipe was 89% busy.
// err: the error bits, then whether queries are left to k_knn_exact.
// Five blocks per SM (a few spills up to k = 4): 7.2 -> 7.05 ms for all eight
// neighbours of 2^22 int64 tuples, 1.57 -> 1.37 for 2^20 float32; six: 7.3, 1.39.
template <typename T, int K>
__global__ void __launch_bounds__(KNN_THREADS, K <= 4 ? 5 : 2) k_knn(const __grid_constant__ KnnTree<T> X,
                                                     const T* __restrict__ queries, int64_t nq, int kn, int width,
                                                     int32_t* __restrict__ idx_out, double* __restrict__ d_out,
                                                     int* __restrict__ err) {
    const int lane = threadIdx.x & 31;
    const int per = 32 / width;
    for (int64_t q0 = ((int64_t)blockIdx.x * (KNN_THREADS / 32) + (threadIdx.x >> 5)) * per; q0 < nq;
         q0 += (int64_t)gridDim.x * (KNN_THREADS / 32) * per) {
        int32_t cand = -1;  // lane r * width + j: candidate j of query q0 + r
        for (int r = 0; r < per && q0 + r < nq; ++r) {
            const int64_t qi = q0 + r;
            KnnQuery<T, K> Q;
            bool nan = false;
#pragma unroll
            for (int d = 0; d < K; ++d) {
                if (K == MAXK && d >= X.k) break;
                Q.q[d] = queries ? queries[qi * (K == MAXK ? X.k : K) + d] : X.pts[d * X.stride + qi];
                nan |= is_nan(Q.q[d]);
            }
            if (nan) {
                if (lane == 0) atomicOr(err, ERR_NAN);
                continue;
            }
            Q.self = queries ? -1 : (int32_t)qi;
            Q.kn = kn;
            Q.bound = KNN_OPEN;
            Q.key = Q.lost = KNN_NONE;
            Q.addr = -1;
            Q.dkey = ~0ull;
            Q.tup = INT32_MAX;
            if (X.m > 0) knn_node<T, K, false, BOX_LEVELS - 1>(X, Q, 0);
            const int32_t c = Q.key != KNN_NONE && Q.key <= Q.bound ? Q.addr : -1;  // the first lanes
            const int cnt = __popc(__ballot_sync(0xffffffffu, c >= 0));
            if (knn_stuck(Q.lost, Q.bound)) {  // left to k_knn_exact
                if (lane == 0) {
                    idx_out[qi * kn] = KNN_LEFT;
                    err[1] = 1;
                }
            } else if (Q.lost <= Q.bound || cnt == 0) {
                // more candidates up to the bound than the list holds, or none at all
                Q.bound = KNN_OPEN;
                if (cnt > 0) knn_node<T, K, true, BOX_LEVELS - 1>(X, Q, 0);
                if (lane < kn) {
                    const bool none = Q.dkey == ~0ull;
                    idx_out[qi * kn + lane] = none ? -1 : Q.tup;
                    if (d_out)
                        d_out[qi * kn + lane] = __longlong_as_double(none ? 0x7ff0000000000000ll : (long long)Q.dkey);
                }
            } else if (cnt > width) {
                knn_emit<T, K>(X, queries, qi, c, 32, kn, idx_out, d_out);
            } else {
                const int32_t v = __shfl_sync(0xffffffffu, c, lane & (width - 1));
                if (lane / width == r) cand = v;
            }
        }
        if (__any_sync(0xffffffffu, cand >= 0))
            knn_emit<T, K>(X, queries, q0 + lane / width, cand, width, kn, idx_out, d_out);
    }
}

// The queries k_knn has left (KNN_LEFT).  Each warp looks at `per` (at most
// 32) rows.
template <typename T, int K>
__global__ void __launch_bounds__(KNN_THREADS, 2) k_knn_exact(const __grid_constant__ KnnTree<T> X,
                                                              const T* __restrict__ queries, int64_t nq, int kn,
                                                              int per, int32_t* __restrict__ idx_out,
                                                              double* __restrict__ d_out) {
    const int lane = threadIdx.x & 31;
    for (int64_t q0 = ((int64_t)blockIdx.x * (KNN_THREADS / 32) + (threadIdx.x >> 5)) * per; q0 < nq;
         q0 += (int64_t)gridDim.x * (KNN_THREADS / 32) * per) {
        const int32_t v = lane < per && q0 + lane < nq ? idx_out[(q0 + lane) * kn] : 0;
        for (uint32_t left = __ballot_sync(0xffffffffu, v == KNN_LEFT); left; left &= left - 1) {
            const int r = __ffs(left) - 1;
            const int64_t qi = q0 + r;
            KnnExact<T, K> Q;
            bool nan = false;
#pragma unroll
            for (int d = 0; d < K; ++d) {
                if (K == MAXK && d >= X.k) break;
                Q.q[d] = queries ? queries[qi * (K == MAXK ? X.k : K) + d] : X.pts[d * X.stride + qi];
                nan |= is_nan(Q.q[d]);
            }
            if (nan) continue;  // (its row was left unwritten, whatever it holds)
            Q.self = queries ? -1 : (int32_t)qi;
            Q.kn = kn;
            Q.last = Q.dkey = ~0ull;
            Q.tup = INT32_MAX;
            knn_exact_node<T, K, BOX_LEVELS - 1>(X, Q, 0);
            if (lane < kn) {
                const bool none = Q.dkey == ~0ull;
                idx_out[qi * kn + lane] = none ? -1 : Q.tup;
                if (d_out)
                    d_out[qi * kn + lane] = __longlong_as_double(none ? 0x7ff0000000000000ll : (long long)Q.dkey);
            }
        }
    }
}

// Boxes of level 0 (src: the point planes, n tuples) or of level l + 1
// (src: the boxes of level l, n of them): one warp per box.
template <typename T>
__global__ void __launch_bounds__(256) k_boxes(const T* __restrict__ src, int64_t stride, int from_points, int64_t n,
                                               int k, int64_t nbox, T* __restrict__ out) {
    const int lane = threadIdx.x & 31;
    for (int64_t b = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5); b < nbox; b += (int64_t)gridDim.x * 8) {
        const int64_t e = b * BOX_W + lane < n ? b * BOX_W + lane : n - 1;  // (a lane past the end repeats the last)
        for (int d = 0; d < k; ++d) {
            T lo, hi;
            if (from_points) {
                lo = hi = src[d * stride + e];
            } else {
                const T* p = src + (e / BOX_W) * (2 * k * BOX_W) + e % BOX_W;
                lo = p[d * BOX_W];
                hi = p[(k + d) * BOX_W];
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const T l2 = __shfl_xor_sync(0xffffffffu, lo, o), h2 = __shfl_xor_sync(0xffffffffu, hi, o);
                lo = l2 < lo ? l2 : lo;
                hi = h2 > hi ? h2 : hi;
            }
            if (lane == 0) {
                T* q = out + (b / BOX_W) * (2 * k * BOX_W) + b % BOX_W;
                q[d * BOX_W] = lo;
                q[(k + d) * BOX_W] = hi;
            }
        }
    }
}

struct KnnEntry {
    int32_t lo, hi, depth;
    double bound;
};

// Insert (d, t) into the sorted list best[0..kn) if it beats the last entry.
__device__ __forceinline__ void knn_insert(double* bd, int32_t* bi, int kn, double d, int32_t t) {
    int j = kn - 1;
    if (!(d < bd[j] || (d == bd[j] && (bi[j] < 0 || t < bi[j])))) return;
    while (j > 0 && (d < bd[j - 1] || (d == bd[j - 1] && (bi[j - 1] < 0 || t < bi[j - 1])))) {
        bd[j] = bd[j - 1];
        bi[j] = bi[j - 1];
        --j;
    }
    bd[j] = d;
    bi[j] = t;
}

// An index without boxes: one thread per query walks the tree depth first,
// near side first.  queries as for k_knn.
template <typename T>
__global__ void __launch_bounds__(SEARCH_THREADS) k_knn_walk(const T* __restrict__ pts, int64_t stride,
                                                             const int32_t* __restrict__ tuple, int32_t m, int k,
                                                             const T* __restrict__ queries, int64_t nq, int kn,
                                                             int32_t* __restrict__ idx_out,
                                                             double* __restrict__ d_out, int* __restrict__ err) {
    const int64_t qi = (int64_t)blockIdx.x * SEARCH_THREADS + threadIdx.x;
    if (qi >= nq) return;
    const int32_t self = queries ? -1 : tuple[qi];
    T q[MAXK];
    bool nan = false;
#pragma unroll
    for (int d = 0; d < MAXK; ++d) {
        q[d] = d < k ? (queries ? queries[qi * k + d] : pts[d * stride + qi]) : (T)0;
        nan |= d < k && is_nan(q[d]);
    }
    if (nan) {
        atomicOr(err, ERR_NAN);
        return;
    }
    double bd[KD_KNN_MAX];
    int32_t bi[KD_KNN_MAX];
    for (int j = 0; j < kn; ++j) {
        bd[j] = __longlong_as_double(0x7ff0000000000000ll);  // +inf
        bi[j] = -1;
    }
    KnnEntry st[STACK_MAX];
    int sp = 0;
    if (m > 0) st[sp++] = KnnEntry{0, m - 1, 0, 0.0};
    while (sp > 0) {
        const KnnEntry e = st[--sp];
        if (e.bound > bd[kn - 1]) continue;  // nothing in this subtree can enter the list
        const int32_t mid = e.lo + ((e.hi - e.lo) >> 1);
        const T* p = pts + mid;
        double acc = 0.0;
        for (int d = 0; d < k; ++d) {
            const double u = abs_diff<T>(p[d * stride], q[d]);
            acc = __dadd_rn(acc, __dmul_rn(u, u));
        }
        const int32_t tm = tuple[mid];
        if (tm != self) knn_insert(bd, bi, kn, acc, tm);
        const int dim = e.depth % k;
        T qd = q[0];
        const T pd = p[dim * stride];
#pragma unroll
        for (int d = 1; d < MAXK; ++d)
            if (d == dim) qd = q[d];
        const double u = abs_diff<T>(pd, qd);
        const double plane = __dmul_rn(u, u);
        const bool less = qd < pd;  // the query lies on the "less" side
        const double far = fmax(e.bound, plane);
        const KnnEntry lo_side{e.lo, mid - 1, e.depth + 1, less ? e.bound : far};
        const KnnEntry hi_side{mid + 1, e.hi, e.depth + 1, less ? far : e.bound};
        if (sp + 2 > STACK_MAX) {
            atomicOr(err, ERR_INTERNAL);
            break;
        }
        // far side below, near side on top
        if (less) {
            if (hi_side.lo <= hi_side.hi) st[sp++] = hi_side;
            if (lo_side.lo <= lo_side.hi) st[sp++] = lo_side;
        } else {
            if (lo_side.lo <= lo_side.hi) st[sp++] = lo_side;
            if (hi_side.lo <= hi_side.hi) st[sp++] = hi_side;
        }
    }
    for (int j = 0; j < kn; ++j) {
        idx_out[qi * kn + j] = bi[j];
        if (d_out) d_out[qi * kn + j] = bd[j];
    }
}

// Boxes in the order of the tree's cells: cell[i] = the segment of level
// `levels` that box i's lower corner falls into, slot[i] its place among the
// cell's boxes so far; then order[] lists the boxes cell by cell.  Walks of
// neighbouring boxes visit the same nodes, so a warp of them diverges less
// and finds them in L1 (the boxes in the caller's order: 21% L1 hits, bound
// by the latency of L2 and DRAM).
template <typename T, int K>
__global__ void __launch_bounds__(256) k_region_cells(const T* __restrict__ pts, int64_t stride, int32_t m, int k,
                                                      int levels, const T* __restrict__ lo, int64_t nq,
                                                      uint32_t* __restrict__ hist, uint32_t* __restrict__ cell,
                                                      uint32_t* __restrict__ slot) {
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= nq) return;
    const int kk = K == MAXK ? k : K;
    T a[K];
#pragma unroll
    for (int d = 0; d < K; ++d)
        if (d < kk) a[d] = lo[i * kk + d];
    int32_t l = 0, h = m - 1;
    uint32_t c = 0;
    for (int lev = 0, dim = 0; lev < levels; ++lev) {
        const int32_t mid = l + ((h - l) >> 1);
        const T p = pts[dim * stride + mid];
        T ad = a[0];
#pragma unroll
        for (int d = 1; d < K; ++d)
            if (d == dim) ad = a[d];
        const bool greater = ad > p;
        c = 2 * c + (greater ? 1u : 0u);
        if (greater) l = mid + 1; else h = mid - 1;
        dim = dim + 1 == kk ? 0 : dim + 1;
    }
    cell[i] = c;
    slot[i] = atomicAdd(&hist[c], 1u);
}
__global__ void __launch_bounds__(256) k_region_order(const uint32_t* __restrict__ cell,
                                                      const uint32_t* __restrict__ slot,
                                                      const int64_t* __restrict__ start, int64_t nq,
                                                      uint32_t* __restrict__ order) {
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (i < nq) order[start[cell[i]] + slot[i]] = (uint32_t)i;
}

// Region search over box qi: count (out == nullptr) or write the indices
// of the tuples inside it at out[offs[qi] ...].  The count may keep the first
// REGION_KEEP of them (kept, row r: the r-th of every box), from which
// k_region_copy then writes the boxes that have no more; the second walk is
// for the others alone (order, *norder of them).  The walk takes a node, its
// less side, then its greater side; the side entered at once stays in
// registers, the other waits on the stack as one word (lo, hi, dimension);
// one kernel per dimension count keeps the box and the node in registers.
// 2^20 boxes of about 3 of 2^22 int64 tuples each: 0.95 -> 0.61 ms a walk, and
// 0.33 with the boxes in cell order.
template <typename T, int K>
__global__ void __launch_bounds__(SEARCH_THREADS) k_region(const T* __restrict__ pts, int64_t stride,
                                                           const int32_t* __restrict__ tuple, int32_t m, int k,
                                                           const T* __restrict__ lo, const T* __restrict__ hi,
                                                           int64_t nq, const uint32_t* __restrict__ order,
                                                           const uint32_t* __restrict__ norder,
                                                           uint32_t* __restrict__ counts, int32_t* __restrict__ kept,
                                                           const int64_t* __restrict__ offs, int32_t* __restrict__ out,
                                                           int* __restrict__ err) {
    const int64_t nwalk = norder ? (int64_t)*norder : nq;
    for (int64_t i = (int64_t)blockIdx.x * SEARCH_THREADS + threadIdx.x; i < nwalk;
         i += (int64_t)gridDim.x * SEARCH_THREADS) {
        const int64_t qi = order ? order[i] : i;
        const int kk = K == MAXK ? k : K;
        T a[K], b[K];
        bool nan = false;
#pragma unroll
        for (int d = 0; d < K; ++d) {
            if (d >= kk) break;
            a[d] = lo[qi * kk + d];
            b[d] = hi[qi * kk + d];
            nan |= is_nan(a[d]) || is_nan(b[d]);
        }
        if (nan) {
            atomicOr(err, ERR_NAN);
            if (!out) counts[qi] = 0;
            continue;
        }
        int64_t o = out ? offs[qi] : 0;
        const int64_t o_end = out ? offs[qi + 1] : 0;
        uint32_t c = 0;
        uint64_t st[REGION_STACK];  // lo | hi << 30 | dimension << 60
        int sp = 0;
        int32_t l = 0, h = m - 1, dim = 0;
        bool more = m > 0;
        while (more) {
            const int32_t mid = l + ((h - l) >> 1);
            T p[K];
#pragma unroll
            for (int d = 0; d < K; ++d)
                if (d < kk) p[d] = pts[d * stride + mid];
            bool in = true, go_less = l < mid, go_greater = mid < h;
#pragma unroll
            for (int d = 0; d < K; ++d) {
                if (d >= kk) break;
                const bool ge = a[d] <= p[d], le = p[d] <= b[d];
                in = in && ge && le;
                if (d == dim) {
                    go_less = go_less && ge;        // the less side holds x_dim <= p_dim
                    go_greater = go_greater && le;  // the greater side holds x_dim >= p_dim
                }
            }
            if (in) {
                if (out) {
                    if (o < o_end) out[o++] = tuple[mid]; else atomicOr(err, ERR_INTERNAL);
                } else if (kept && c < (uint32_t)REGION_KEEP) {
                    kept[(int64_t)c * nq + qi] = tuple[mid];
                }
                ++c;
            }
            dim = dim + 1 == kk ? 0 : dim + 1;
            if (go_less) {
                if (go_greater) {
                    if (sp == REGION_STACK) {
                        atomicOr(err, ERR_INTERNAL);
                        break;
                    }
                    st[sp++] = (uint64_t)(uint32_t)(mid + 1) | ((uint64_t)(uint32_t)h << 30) | ((uint64_t)dim << 60);
                }
                h = mid - 1;
            } else if (go_greater) {
                l = mid + 1;
            } else if (sp > 0) {
                const uint64_t e = st[--sp];
                l = (int32_t)(e & 0x3fffffffu);
                h = (int32_t)((e >> 30) & 0x3fffffffu);
                dim = (int)(e >> 60);
            } else {
                more = false;
            }
        }
        if (!out) counts[qi] = c;
    }
}

// Writes the boxes of at most REGION_KEEP tuples from kept and lists the
// others.
__global__ void __launch_bounds__(256) k_region_copy(const uint32_t* __restrict__ counts,
                                                     const int64_t* __restrict__ offs,
                                                     const int32_t* __restrict__ kept, int64_t nq,
                                                     int32_t* __restrict__ out, uint32_t* __restrict__ list,
                                                     uint32_t* __restrict__ nlist) {
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    const uint32_t c = i < nq ? counts[i] : 0u;
    const bool many = c > (uint32_t)REGION_KEEP;
    const uint32_t b = __ballot_sync(0xffffffffu, many);
    if (b) {
        const int lane = threadIdx.x & 31, first = __ffs(b) - 1;
        uint32_t at = 0;
        if (lane == first) at = atomicAdd(nlist, (uint32_t)__popc(b));
        at = __shfl_sync(0xffffffffu, at, first);
        if (many) list[at + __popc(b & kd::lanemask_lt())] = (uint32_t)i;
    }
    if (many || c == 0) return;
    const int64_t o = offs[i];
#pragma unroll
    for (uint32_t r = 0; r < (uint32_t)REGION_KEEP; ++r)
        if (r < c) out[o + r] = kept[(int64_t)r * nq + i];
}

// Reverse nearest neighbours: inv[tuple] = address, then per target
// address the number of nodes listing it, then the lists.
__global__ void __launch_bounds__(256) k_inv_map(const int32_t* __restrict__ tuple, int64_t m, int64_t n,
                                                 int32_t* __restrict__ inv, int* __restrict__ err) {
    for (int64_t a = (int64_t)blockIdx.x * 256 + threadIdx.x; a < m; a += (int64_t)gridDim.x * 256) {
        const int32_t t = tuple[a];
        if (t < 0 || t >= n) atomicOr(err, ERR_INTERNAL); else inv[t] = (int32_t)a;
    }
}
__global__ void __launch_bounds__(256) k_rev_count(const int32_t* __restrict__ nn, int64_t total,
                                                   const int32_t* __restrict__ inv, int64_t n,
                                                   int64_t* __restrict__ cnt, int* __restrict__ err) {
    for (int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x; e < total; e += (int64_t)gridDim.x * 256) {
        const int32_t t = nn[e];
        if (t < 0) continue;
        const int32_t a = t < n ? inv[t] : -1;
        if (a < 0) atomicOr(err, ERR_INTERNAL); else atomicAdd((unsigned long long*)&cnt[a], 1ull);
    }
}
__global__ void __launch_bounds__(256) k_rev_fill(const int32_t* __restrict__ nn, int64_t total, int kn,
                                                  const int32_t* __restrict__ tuple, const int32_t* __restrict__ inv,
                                                  int64_t n, int64_t* __restrict__ cursor, int32_t* __restrict__ rev,
                                                  int* __restrict__ err) {
    for (int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x; e < total; e += (int64_t)gridDim.x * 256) {
        const int32_t t = nn[e];
        if (t < 0) continue;
        const int32_t a = t < n ? inv[t] : -1;
        if (a < 0) {
            atomicOr(err, ERR_INTERNAL);
            continue;
        }
        const int64_t pos = (int64_t)atomicAdd((unsigned long long*)&cursor[a], 1ull);
        rev[pos] = tuple[e / kn];
    }
}

// offs[i] = sum of counts[0..i), offs[n] = total, in three launches: the
// sum of every chunk of OFF_CHUNK counts, their exclusive scan by one block,
// and every chunk's own scan from its base.  (One block scanning all counts
// 1024 at a time took 1.08 ms for 2^20 of them: a serial chain of barriers
// on one SM.)
constexpr int OFF_VPT = 8;
constexpr int OFF_CHUNK = 256 * OFF_VPT;

// Inclusive scan of one value per lane.
__device__ __forceinline__ int64_t warp_incl(int64_t x) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    return x;
}

template <typename C>
__global__ void __launch_bounds__(256) k_offsets_sums(const C* __restrict__ counts, int64_t n,
                                                      int64_t* __restrict__ sums) {
    __shared__ int64_t s_w[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int64_t v = 0;
#pragma unroll
    for (int j = 0; j < OFF_VPT; ++j) {
        const int64_t i = (int64_t)blockIdx.x * OFF_CHUNK + j * 256 + threadIdx.x;
        v += i < n ? (int64_t)counts[i] : 0;
    }
    v = warp_incl(v);
    if (lane == 31) s_w[warp] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        int64_t t = 0;
        for (int w = 0; w < 8; ++w) t += s_w[w];
        sums[blockIdx.x] = t;
    }
}

__global__ void __launch_bounds__(1024) k_offsets_bases(int64_t nchunks, int64_t* __restrict__ sums,
                                                        int64_t* __restrict__ total) {
    __shared__ int64_t s_w[32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int64_t carry = 0;
    for (int64_t base = 0; base < nchunks; base += 1024) {
        const int64_t i = base + tid;
        const int64_t v = i < nchunks ? sums[i] : 0;
        const int64_t x = warp_incl(v);
        if (lane == 31) s_w[warp] = x;
        __syncthreads();
        if (warp == 0) s_w[lane] = warp_incl(s_w[lane]);
        __syncthreads();
        if (i < nchunks) sums[i] = carry + (warp ? s_w[warp - 1] : 0) + x - v;
        carry += s_w[31];
        __syncthreads();
    }
    if (tid == 0) *total = carry;
}

template <typename C>
__global__ void __launch_bounds__(256) k_offsets_write(const C* __restrict__ counts, int64_t n,
                                                       const int64_t* __restrict__ sums, int64_t* __restrict__ offs) {
    __shared__ int64_t s_w[OFF_VPT][8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t base = (int64_t)blockIdx.x * OFF_CHUNK;
    int64_t v[OFF_VPT], x[OFF_VPT];
#pragma unroll
    for (int j = 0; j < OFF_VPT; ++j) {
        const int64_t i = base + j * 256 + threadIdx.x;
        v[j] = i < n ? (int64_t)counts[i] : 0;
    }
#pragma unroll
    for (int j = 0; j < OFF_VPT; ++j) {
        x[j] = warp_incl(v[j]);
        if (lane == 31) s_w[j][warp] = x[j];
    }
    __syncthreads();
    int64_t run = sums[blockIdx.x];
#pragma unroll
    for (int j = 0; j < OFF_VPT; ++j) {
        int64_t before = run;
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            if (w < warp) before += s_w[j][w];
            run += s_w[j][w];
        }
        const int64_t i = base + j * 256 + threadIdx.x;
        if (i < n) offs[i] = before + x[j] - v[j];
    }
}

size_t dtype_size(int dtype) { return dtype == KD_I64 ? 8 : 4; }

kd_status sfail(kd_ctx* ctx, kd_status code, const std::string& msg) {
    kd::ctx_set_error(ctx, msg);
    return code;
}

// Scratch owned by one call.
struct CallScratch {
    kd_ctx* ctx;
    std::vector<void*> ptrs;
    explicit CallScratch(kd_ctx* c) : ctx(c) {}
    ~CallScratch() { clear(); }
    void clear() {
        for (void* p : ptrs) kd::ctx_free(ctx, p);
        ptrs.clear();
    }
    kd_status get(void** p, size_t bytes) {
        kd_status s = kd::ctx_alloc(ctx, p, bytes);
        if (s == KD_OK) ptrs.push_back(*p);
        return s;
    }
};

// A device copy of host data (or the device pointer itself).
kd_status to_device(kd_ctx* ctx, CallScratch& S, const void* src, size_t bytes, int on_device, const void** out,
                    cudaStream_t s) {
    if (on_device || bytes == 0) {
        *out = src;
        return KD_OK;
    }
    void* d = nullptr;
    kd_status st = S.get(&d, bytes);
    if (st != KD_OK) return st;
    if (cudaMemcpyAsync(d, src, bytes, cudaMemcpyHostToDevice, s) != cudaSuccess)
        return sfail(ctx, KD_EDEVICE, "host to device copy failed");
    *out = d;
    return KD_OK;
}

// The error word after everything on the stream; left (if given): the word
// after it.
kd_status read_err(kd_ctx* ctx, int* d_err, cudaStream_t s, int* left = nullptr) {
    int words[2] = {0, 0};
    if (cudaMemcpyAsync(words, d_err, (left ? 2 : 1) * sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return sfail(ctx, KD_EDEVICE, std::string("search: ") + cudaGetErrorString(cudaGetLastError()));
    const int h = words[0];
    if (left) *left = words[1];
    if (h & ERR_NAN) return sfail(ctx, KD_ENAN, "a query coordinate is NaN");
    if (h) return sfail(ctx, KD_EDEVICE, "inconsistent tree or index (device error flags " + std::to_string(h) + ")");
    return KD_OK;
}

int grid_of(int64_t n, int per) { return (int)std::max<int64_t>(1, std::min<int64_t>((n + per - 1) / per, 1 << 20)); }

// Levels of boxes over m tuples: words per level (whole groups of 32
// siblings) and in all; returns the total.
int64_t box_layout(kd_index_s* ix) {
    int64_t words = 0, n = ix->m;
    for (int l = 0; l < BOX_LEVELS; ++l) {
        n = (n + BOX_W - 1) / BOX_W;
        ix->nbox[l] = (int32_t)n;
        ix->box_off[l] = words;
        words += (n + BOX_W - 1) / BOX_W * (2 * ix->k * BOX_W);
        ix->top = l;
        if (n <= BOX_W) break;
    }
    return words;
}

// The planes and boxes of a new index from coords and the tree.
template <typename T>
void index_fill(kd_ctx* ctx, kd_index_s* ix, const void* coords, int64_t n, int* err, cudaStream_t s) {
    k_index_gather<T><<<grid_of(ix->m, 256), 256, 0, s>>>((const T*)coords, ix->node_tuple, ix->m, ix->k, n,
                                                          (T*)ix->pts, err);
    kd::ctx_add_launches(ctx, 1);
    if (!ix->boxes) return;
    for (int l = 0; l <= ix->top; ++l) {
        const T* src = l ? (const T*)ix->boxes + ix->box_off[l - 1] : (const T*)ix->pts;
        k_boxes<T><<<grid_of(ix->nbox[l], 8), 256, 0, s>>>(src, ix->m, l == 0, l ? ix->nbox[l - 1] : ix->m, ix->k,
                                                           ix->nbox[l], (T*)ix->boxes + ix->box_off[l]);
        kd::ctx_add_launches(ctx, 1);
    }
}

// Whether the m tuples of a plane fill at least a quarter of the integer points
// of their range, from the top level's boxes (b: one group, on the host).
template <typename T>
bool index_dense(const kd_index_s* ix, const T* b) {
    double points = 1.0;
    for (int d = 0; d < 2; ++d) {
        const T lo = *std::min_element(b + d * BOX_W, b + d * BOX_W + ix->nbox[ix->top]);
        const T hi = *std::max_element(b + (2 + d) * BOX_W, b + (2 + d) * BOX_W + ix->nbox[ix->top]);
        points *= (double)hi - (double)lo + 1.0;
    }
    return points <= 4.0 * (double)ix->m;
}

template <typename T, int K>
void knn_as(kd_index_s* ix, const void* queries, int64_t nq, int kn, int32_t* di, double* dd, int* err, bool exact,
            cudaStream_t s) {
    KnnTree<T> X{};
    X.pts = (const T*)ix->pts;
    X.stride = ix->m;
    X.tuple = ix->node_tuple;
    X.m = (int32_t)ix->m;
    X.k = ix->k;
    X.top = ix->top;
    for (int l = 0; l <= ix->top; ++l) {
        X.box[l] = (const T*)ix->boxes + ix->box_off[l];
        X.nbox[l] = ix->nbox[l];
    }
    if (exact) {
        const int per = (int)std::max<int64_t>(1, std::min<int64_t>(32, nq / (152 * 32 * 4)));
        k_knn_exact<T, K><<<grid_of(nq, KNN_THREADS / 32 * per), KNN_THREADS, 0, s>>>(X, (const T*)queries, nq, kn, per,
                                                                                     di, dd);
        return;
    }
    // several queries per warp only where there are warps enough without it (152 SMs x 32 warps)
    int width = 32;
    while (width / 2 >= kn && width > 4 && nq * width / 64 >= 152 * 32) width /= 2;
    const int per = KNN_THREADS / width;  // queries of a block at a time
    k_knn<T, K><<<grid_of(nq, per), KNN_THREADS, 0, s>>>(X, (const T*)queries, nq, kn, width, di, dd, err);
}

template <typename T, int K>
void region_as(kd_index_s* ix, const void* lo, const void* hi, int64_t nq, const uint32_t* order,
               const uint32_t* norder, uint32_t* counts, int32_t* kept, const int64_t* offs, int32_t* out, int* err,
               cudaStream_t s) {
    k_region<T, K><<<grid_of(nq, SEARCH_THREADS), SEARCH_THREADS, 0, s>>>(
        (const T*)ix->pts, ix->m, ix->node_tuple, (int32_t)ix->m, ix->k, (const T*)lo, (const T*)hi, nq, order, norder,
        counts, kept, offs, out, err);
}

template <typename T, int K>
void cells_as(kd_index_s* ix, int levels, const void* lo, int64_t nq, uint32_t* hist, uint32_t* cell, uint32_t* slot,
              cudaStream_t s) {
    k_region_cells<T, K><<<(unsigned)((nq + 255) / 256), 256, 0, s>>>((const T*)ix->pts, ix->m, (int32_t)ix->m, ix->k,
                                                                      levels, (const T*)lo, nq, hist, cell, slot);
}

// Calls NAME<T, K>(...): K the index's dimension count, MAXK for those
// without kernels of their own.
#define KD_SEARCH_K(NAME, T, ...)                                 \
    switch (ix->k) {                                              \
        case 2: NAME<T, 2>(__VA_ARGS__); break;                   \
        case 3: NAME<T, 3>(__VA_ARGS__); break;                   \
        case 4: NAME<T, 4>(__VA_ARGS__); break;                   \
        default: NAME<T, MAXK>(__VA_ARGS__); break;               \
    }

// Searches of few neighbours that one thread each answers faster than one warp
// each: over one dimension, whose split planes are its distances, or over a
// plane whose points fill it, where the boxes touch and tie.  One nearest and
// two nearest of each of 2^20 tuples, by warps and by threads: k = 1 int32 0.92
// and 0.66, 0.93 and 0.74 ms (four nearest 0.97 and 0.96, of half-filled
// integers 0.87 and 0.75, of float32 1.09 and 1.19; 4096 tuples 0.05 and 0.09),
// a half-filled lattice of k = 2 1.84 and 1.38, 2.04 and 1.58 (four nearest 2.40
// and 2.00; eight 0.36 and 0.49 at 2^17), spread int32 of k = 2 0.68 and 1.49.
constexpr int64_t WALK_MIN_QUERIES = 1 << 16;
bool knn_by_walk(const kd_index_s* ix, int64_t nq, int kn) {
    if (!ix->boxes) return true;
    return nq >= WALK_MIN_QUERIES && (ix->k == 1 || ix->dense) && kn <= (ix->dtype == KD_F32 ? 2 : 4);
}

template <typename T>
void knn_of(kd_index_s* ix, const void* queries, int64_t nq, int kn, int32_t* di, double* dd, int* err, bool exact,
            cudaStream_t s) {
    if (ix->m > 0 && knn_by_walk(ix, nq, kn))  // (a thread per query, so a grid that no cap of grid_of cuts)
        k_knn_walk<T><<<(unsigned)((nq + SEARCH_THREADS - 1) / SEARCH_THREADS), SEARCH_THREADS, 0, s>>>(
            (const T*)ix->pts, ix->m, ix->node_tuple, (int32_t)ix->m, ix->k, (const T*)queries, nq, kn, di, dd, err);
    else
        KD_SEARCH_K(knn_as, T, ix, queries, nq, kn, di, dd, err, exact, s)
}

// The kn nearest tuples of nq queries (nullptr: of every address); exact: of
// those of them that such a call has left (err[1], which it sets).
void launch_knn(kd_ctx* ctx, kd_index_s* ix, const void* queries, int64_t nq, int kn, int32_t* di, double* dd,
                int* err, bool exact, cudaStream_t s) {
    if (ix->dtype == KD_I32) knn_of<int32_t>(ix, queries, nq, kn, di, dd, err, exact, s);
    else if (ix->dtype == KD_I64) knn_of<int64_t>(ix, queries, nq, kn, di, dd, err, exact, s);
    else knn_of<float>(ix, queries, nq, kn, di, dd, err, exact, s);
    kd::ctx_add_launches(ctx, 1);
}

void launch_region(kd_ctx* ctx, kd_index_s* ix, const void* lo, const void* hi, int64_t nq, const uint32_t* order,
                   const uint32_t* norder, uint32_t* counts, int32_t* kept, const int64_t* offs, int32_t* out, int* err,
                   cudaStream_t s) {
    if (nq == 0) return;
    if (ix->dtype == KD_I32) KD_SEARCH_K(region_as, int32_t, ix, lo, hi, nq, order, norder, counts, kept, offs, out, err, s)
    else if (ix->dtype == KD_I64) KD_SEARCH_K(region_as, int64_t, ix, lo, hi, nq, order, norder, counts, kept, offs, out, err, s)
    else KD_SEARCH_K(region_as, float, ix, lo, hi, nq, order, norder, counts, kept, offs, out, err, s)
    kd::ctx_add_launches(ctx, 1);
}

// launch_knn with the copies of host outputs, to its end; once more for the
// queries it has left, if any.
kd_status run_knn(kd_ctx* ctx, kd_index_s* ix, const void* queries, int64_t nq, int kn, int32_t* di, double* dd,
                  int* d_err, int on_device, int32_t* idx_out, double* dist_out, cudaStream_t s) {
    for (bool exact = false;; exact = true) {
        launch_knn(ctx, ix, queries, nq, kn, di, dd, d_err, exact, s);
        if (!on_device) {
            cudaMemcpyAsync(idx_out, di, (size_t)nq * kn * 4, cudaMemcpyDeviceToHost, s);
            if (dist_out) cudaMemcpyAsync(dist_out, dd, (size_t)nq * kn * 8, cudaMemcpyDeviceToHost, s);
        }
        int left = 0;
        const kd_status st = read_err(ctx, d_err, s, &left);
        if (exact || !left || (st != KD_OK && st != KD_ENAN)) return st;
    }
}

int64_t offsets_chunks(int64_t n) { return std::max<int64_t>(1, (n + OFF_CHUNK - 1) / OFF_CHUNK); }

// offs[0..n] from counts[0..n); sums: offsets_chunks(n) words.
template <typename C>
void launch_offsets(kd_ctx* ctx, const C* counts, int64_t n, int64_t* sums, int64_t* offs, cudaStream_t s) {
    const int64_t chunks = offsets_chunks(n);
    k_offsets_sums<C><<<(unsigned)chunks, 256, 0, s>>>(counts, n, sums);
    k_offsets_bases<<<1, 1024, 0, s>>>(chunks, sums, offs + n);
    k_offsets_write<C><<<(unsigned)chunks, 256, 0, s>>>(counts, n, sums, offs);
    kd::ctx_add_launches(ctx, 3);
}

// The boxes' order (nullptr: the caller's, for few boxes or tuples, or where
// the workspace does not fit).  Counting and writing 2^20 boxes in 2^22
// int64 tuples: 1.96 ms in the caller's order, 1.40 cell by cell; 2^17 boxes
// 0.55 and 0.54, 2^15 0.39 and 0.43 (its launches cost more than it gains).
constexpr int CELL_LEVELS = 14;
constexpr int64_t CELL_MIN_BOXES = 1 << 17;
// Boxes from which the count keeps their first tuples: 2^20 boxes 1.41 -> 1.28
// ms, 2^17 boxes 0.54 -> 0.60.
constexpr int64_t KEEP_MIN_BOXES = 1 << 19;
const uint32_t* region_order(kd_ctx* ctx, kd_index_s* ix, CallScratch& S, const void* lo, int64_t nq, cudaStream_t s) {
    if (nq < CELL_MIN_BOXES || nq > UINT32_MAX || ix->m < (1 << 16)) return nullptr;
    int levels = 0;
    while (levels < CELL_LEVELS && (ix->m >> (levels + 4)) > 0) ++levels;
    const int64_t cells = (int64_t)1 << levels, chunks = offsets_chunks(cells);
    unsigned char* w = nullptr;
    if (S.get((void**)&w, (size_t)(cells + 1 + chunks) * 8 + (size_t)(cells + 3 * nq) * 4) != KD_OK) {
        sfail(ctx, KD_OK, "");
        return nullptr;
    }
    int64_t* start = (int64_t*)w;
    int64_t* sums = start + cells + 1;
    uint32_t* hist = (uint32_t*)(sums + chunks);
    uint32_t *cell = hist + cells, *slot = cell + nq, *order = slot + nq;
    cudaMemsetAsync(hist, 0, (size_t)cells * 4, s);
    if (ix->dtype == KD_I32) KD_SEARCH_K(cells_as, int32_t, ix, levels, lo, nq, hist, cell, slot, s)
    else if (ix->dtype == KD_I64) KD_SEARCH_K(cells_as, int64_t, ix, levels, lo, nq, hist, cell, slot, s)
    else KD_SEARCH_K(cells_as, float, ix, levels, lo, nq, hist, cell, slot, s)
    launch_offsets(ctx, hist, cells, sums, start, s);
    k_region_order<<<(unsigned)((nq + 255) / 256), 256, 0, s>>>(cell, slot, start, nq, order);
    kd::ctx_add_launches(ctx, 2);
    return order;
}

}  // namespace

extern "C" {

kd_status kd_index_create(kd_ctx* ctx, const kd_cloud* cloud, const kd_tree* tree, kd_index* out) {
    if (!ctx || !out) return KD_EINVAL;
    *out = nullptr;
    std::lock_guard<std::recursive_mutex> lk(kd::ctx_mutex(ctx));
    if (cudaSetDevice(kd::ctx_device(ctx)) != cudaSuccess) return sfail(ctx, KD_EDEVICE, "cudaSetDevice failed");
    if (!cloud || !tree) return sfail(ctx, KD_EINVAL, "cloud or tree is NULL");
    if (cloud->k < 1 || cloud->k > KD_MAX_K || cloud->n < 0 || cloud->n > KD_MAX_N ||
        (cloud->dtype != KD_I32 && cloud->dtype != KD_I64 && cloud->dtype != KD_F32))
        return sfail(ctx, KD_EINVAL, "bad cloud");
    if (tree->m < 0 || tree->m > cloud->n || (tree->m > 0 && (!tree->node_tuple || !cloud->coords)))
        return sfail(ctx, KD_EINVAL, "tree does not fit the cloud");
    cudaStream_t s = kd::ctx_stream(ctx);
    const size_t ts = dtype_size(cloud->dtype);
    std::unique_ptr<kd_index_s> ix(new kd_index_s());
    ix->ctx = ctx;
    ix->m = tree->m;
    ix->k = cloud->k;
    ix->dtype = cloud->dtype;
    if (ix->m == 0) {
        *out = ix.release();
        return KD_OK;
    }
    CallScratch S(ctx);
    const void* coords = nullptr;
    const void* tuple = nullptr;
    kd_status st = to_device(ctx, S, cloud->coords, (size_t)cloud->n * cloud->k * ts, cloud->on_device, &coords, s);
    if (st == KD_OK) st = to_device(ctx, S, tree->node_tuple, (size_t)ix->m * 4, tree->on_device, &tuple, s);
    if (st == KD_OK) st = kd::ctx_alloc(ctx, &ix->pts, (size_t)ix->m * ix->k * ts);
    if (st == KD_OK) st = kd::ctx_alloc(ctx, (void**)&ix->node_tuple, (size_t)ix->m * 4);
    int* d_err = nullptr;
    if (st == KD_OK) st = S.get((void**)&d_err, sizeof(int));
    if (st != KD_OK) {
        kd_index_destroy(ctx, ix.release());
        return st;
    }
    // the boxes (a sixteenth of the planes) are left out where they do not fit the budget
    if (kd::ctx_alloc(ctx, &ix->boxes, (size_t)box_layout(ix.get()) * ts) != KD_OK) sfail(ctx, KD_OK, "");
    cudaMemsetAsync(d_err, 0, sizeof(int), s);
    cudaMemcpyAsync(ix->node_tuple, tuple, (size_t)ix->m * 4, cudaMemcpyDeviceToDevice, s);
    if (ix->dtype == KD_I32) index_fill<int32_t>(ctx, ix.get(), coords, cloud->n, d_err, s);
    else if (ix->dtype == KD_I64) index_fill<int64_t>(ctx, ix.get(), coords, cloud->n, d_err, s);
    else index_fill<float>(ctx, ix.get(), coords, cloud->n, d_err, s);
    const bool plane = ix->boxes && ix->k == 2 && ix->dtype != KD_F32;
    int64_t range[4 * BOX_W];
    if (plane)
        cudaMemcpyAsync(range, (const char*)ix->boxes + ix->box_off[ix->top] * ts, 4 * BOX_W * ts,
                        cudaMemcpyDeviceToHost, s);
    st = read_err(ctx, d_err, s);
    if (st != KD_OK) {
        kd_index_destroy(ctx, ix.release());
        return st;
    }
    if (plane)
        ix->dense = ix->dtype == KD_I32 ? index_dense(ix.get(), reinterpret_cast<const int32_t*>(range))
                                        : index_dense(ix.get(), range);
    *out = ix.release();
    return KD_OK;
}

kd_status kd_index_destroy(kd_ctx* ctx, kd_index ix) {
    if (!ctx || !ix) return KD_EINVAL;
    std::lock_guard<std::recursive_mutex> lk(kd::ctx_mutex(ctx));
    cudaSetDevice(kd::ctx_device(ctx));
    if (ix->pts) kd::ctx_free(ctx, ix->pts);
    if (ix->boxes) kd::ctx_free(ctx, ix->boxes);
    if (ix->node_tuple) kd::ctx_free(ctx, ix->node_tuple);
    delete ix;
    return KD_OK;
}

kd_status kd_knn(kd_ctx* ctx, kd_index ix, const void* queries, int64_t nq, int kn, int on_device, int32_t* idx_out,
                 double* dist_out) {
    if (!ctx || !ix) return KD_EINVAL;
    std::lock_guard<std::recursive_mutex> lk(kd::ctx_mutex(ctx));
    if (cudaSetDevice(kd::ctx_device(ctx)) != cudaSuccess) return sfail(ctx, KD_EDEVICE, "cudaSetDevice failed");
    if (kn < 1 || kn > KD_KNN_MAX) return sfail(ctx, KD_EINVAL, "kn must be in [1, KD_KNN_MAX]");
    if (nq < 0 || (nq > 0 && (!queries || !idx_out))) return sfail(ctx, KD_EINVAL, "bad queries or outputs");
    if (nq == 0) return KD_OK;
    cudaStream_t s = kd::ctx_stream(ctx);
    const size_t ts = dtype_size(ix->dtype);
    CallScratch S(ctx);
    const void* q = nullptr;
    kd_status st = to_device(ctx, S, queries, (size_t)nq * ix->k * ts, on_device, &q, s);
    int32_t* di = idx_out;
    double* dd = dist_out;
    int* d_err = nullptr;
    if (st == KD_OK && !on_device) {
        st = S.get((void**)&di, (size_t)nq * kn * 4);
        if (st == KD_OK && dist_out) st = S.get((void**)&dd, (size_t)nq * kn * 8);
    }
    if (st == KD_OK) st = S.get((void**)&d_err, 2 * sizeof(int));
    if (st != KD_OK) return st;
    cudaMemsetAsync(d_err, 0, 2 * sizeof(int), s);
    return run_knn(ctx, ix, q, nq, kn, di, dd, d_err, on_device, idx_out, dist_out, s);
}

kd_status kd_knn_all(kd_ctx* ctx, kd_index ix, int kn, int on_device, int32_t* idx_out, double* dist_out) {
    if (!ctx || !ix) return KD_EINVAL;
    std::lock_guard<std::recursive_mutex> lk(kd::ctx_mutex(ctx));
    if (cudaSetDevice(kd::ctx_device(ctx)) != cudaSuccess) return sfail(ctx, KD_EDEVICE, "cudaSetDevice failed");
    if (kn < 1 || kn > KD_KNN_MAX) return sfail(ctx, KD_EINVAL, "kn must be in [1, KD_KNN_MAX]");
    if (ix->m > 0 && !idx_out) return sfail(ctx, KD_EINVAL, "idx_out is NULL");
    if (ix->m == 0) return KD_OK;
    cudaStream_t s = kd::ctx_stream(ctx);
    CallScratch S(ctx);
    int32_t* di = idx_out;
    double* dd = dist_out;
    int* d_err = nullptr;
    kd_status st = KD_OK;
    if (!on_device) {
        st = S.get((void**)&di, (size_t)ix->m * kn * 4);
        if (st == KD_OK && dist_out) st = S.get((void**)&dd, (size_t)ix->m * kn * 8);
    }
    if (st == KD_OK) st = S.get((void**)&d_err, 2 * sizeof(int));
    if (st != KD_OK) return st;
    cudaMemsetAsync(d_err, 0, 2 * sizeof(int), s);
    return run_knn(ctx, ix, nullptr, ix->m, kn, di, dd, d_err, on_device, idx_out, dist_out, s);
}

kd_status kd_reverse_knn(kd_ctx* ctx, kd_index ix, int kn, int on_device, int64_t* offsets, int32_t* rev_out) {
    if (!ctx || !ix) return KD_EINVAL;
    std::lock_guard<std::recursive_mutex> lk(kd::ctx_mutex(ctx));
    if (cudaSetDevice(kd::ctx_device(ctx)) != cudaSuccess) return sfail(ctx, KD_EDEVICE, "cudaSetDevice failed");
    if (kn < 1 || kn > KD_KNN_MAX) return sfail(ctx, KD_EINVAL, "kn must be in [1, KD_KNN_MAX]");
    if (!offsets || (ix->m > 0 && !rev_out)) return sfail(ctx, KD_EINVAL, "offsets or rev_out is NULL");
    cudaStream_t s = kd::ctx_stream(ctx);
    const int64_t m = ix->m, total = m * kn;
    CallScratch S(ctx);
    int32_t *nn = nullptr, *inv = nullptr, *rev = rev_out;
    int64_t *cnt = nullptr, *offs = offsets, *cursor = nullptr;
    int* d_err = nullptr;
    int64_t n = 0;  // tuple indices are below the largest one + 1; the inverse map spans them
    kd_status st = S.get((void**)&d_err, 2 * sizeof(int));
    if (st != KD_OK) return st;
    if (m == 0) {
        int64_t z = 0;
        if (on_device) cudaMemcpyAsync(offsets, &z, 8, cudaMemcpyHostToDevice, s); else offsets[0] = 0;
        return cudaStreamSynchronize(s) == cudaSuccess ? KD_OK : sfail(ctx, KD_EDEVICE, "synchronise failed");
    }
    // the inverse map needs the largest tuple index
    {
        std::vector<int32_t> tmp;
        int32_t mx = 0;
        tmp.resize((size_t)m);
        if (cudaMemcpyAsync(tmp.data(), ix->node_tuple, (size_t)m * 4, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            cudaStreamSynchronize(s) != cudaSuccess)
            return sfail(ctx, KD_EDEVICE, "reading the index failed");
        for (int32_t t : tmp) mx = std::max(mx, t);
        n = (int64_t)mx + 1;
    }
    st = S.get((void**)&nn, (size_t)total * 4);
    if (st == KD_OK) st = S.get((void**)&inv, (size_t)n * 4);
    if (st == KD_OK) st = S.get((void**)&cnt, (size_t)m * 8);
    if (st == KD_OK) st = S.get((void**)&cursor, (size_t)(m + 1) * 8);
    if (st == KD_OK && !on_device) {
        st = S.get((void**)&offs, (size_t)(m + 1) * 8);
        if (st == KD_OK) st = S.get((void**)&rev, (size_t)std::max<int64_t>(total, 1) * 4);
    }
    if (st != KD_OK) return st;
    cudaMemsetAsync(d_err, 0, 2 * sizeof(int), s);
    cudaMemsetAsync(inv, 0xff, (size_t)n * 4, s);
    cudaMemsetAsync(cnt, 0, (size_t)m * 8, s);
    launch_knn(ctx, ix, nullptr, m, kn, nn, nullptr, d_err, false, s);
    if (!knn_by_walk(ix, m, kn))
        launch_knn(ctx, ix, nullptr, m, kn, nn, nullptr, d_err, true, s);  // (finds none to do, mostly)
    k_inv_map<<<grid_of(m, 256), 256, 0, s>>>(ix->node_tuple, m, n, inv, d_err);
    k_rev_count<<<grid_of(total, 256), 256, 0, s>>>(nn, total, inv, n, cnt, d_err);
    launch_offsets(ctx, cnt, m, cursor, offs, s);  // (the cursors' words hold the chunk sums meanwhile)
    cudaMemcpyAsync(cursor, offs, (size_t)(m + 1) * 8, cudaMemcpyDeviceToDevice, s);
    k_rev_fill<<<grid_of(total, 256), 256, 0, s>>>(nn, total, kn, ix->node_tuple, inv, n, cursor, rev, d_err);
    kd::ctx_add_launches(ctx, 3);
    int64_t tot = 0;
    cudaMemcpyAsync(&tot, offs + m, 8, cudaMemcpyDeviceToHost, s);
    if (!on_device) {
        cudaMemcpyAsync(offsets, offs, (size_t)(m + 1) * 8, cudaMemcpyDeviceToHost, s);
        cudaMemcpyAsync(rev_out, rev, (size_t)total * 4, cudaMemcpyDeviceToHost, s);
    }
    return read_err(ctx, d_err, s);
}

kd_status kd_region(kd_ctx* ctx, kd_index ix, const void* lo, const void* hi, int64_t nq, int on_device,
                    int64_t* offsets, int32_t* idx_out, int64_t capacity) {
    if (!ctx || !ix) return KD_EINVAL;
    std::lock_guard<std::recursive_mutex> lk(kd::ctx_mutex(ctx));
    if (cudaSetDevice(kd::ctx_device(ctx)) != cudaSuccess) return sfail(ctx, KD_EDEVICE, "cudaSetDevice failed");
    if (nq < 0 || !offsets || (nq > 0 && (!lo || !hi))) return sfail(ctx, KD_EINVAL, "bad boxes or offsets");
    cudaStream_t s = kd::ctx_stream(ctx);
    const size_t ts = dtype_size(ix->dtype);
    CallScratch S(ctx);
    const void *dlo = nullptr, *dhi = nullptr;
    kd_status st = to_device(ctx, S, lo, (size_t)nq * ix->k * ts, on_device, &dlo, s);
    if (st == KD_OK) st = to_device(ctx, S, hi, (size_t)nq * ix->k * ts, on_device, &dhi, s);
    uint32_t* counts = nullptr;
    int64_t *sums = nullptr, *doffs = offsets;
    int* d_err = nullptr;
    const int64_t chunks = offsets_chunks(nq);  // the chunk sums of the scan, then the counts, in one allocation
    if (st == KD_OK) st = S.get((void**)&sums, (size_t)chunks * 8 + (size_t)nq * 4);
    counts = reinterpret_cast<uint32_t*>(sums + chunks);
    if (st == KD_OK && !on_device) st = S.get((void**)&doffs, (size_t)(nq + 1) * 8);
    if (st == KD_OK) st = S.get((void**)&d_err, sizeof(int));
    if (st != KD_OK) return st;
    cudaMemsetAsync(d_err, 0, sizeof(int), s);
    CallScratch O(ctx);  // what the walks only go faster with
    const uint32_t* order = region_order(ctx, ix, O, dlo, nq, s);
    // where the indices of many boxes are wanted, the first of every box are
    // kept (if they fit), then the list of the boxes that have more and its
    // length.  (Of few boxes, some have more, and the second walk takes as
    // long for them as for all.)
    int32_t* kept = nullptr;
    if (idx_out && nq >= KEEP_MIN_BOXES && nq <= UINT32_MAX &&
        O.get((void**)&kept, ((size_t)nq * (REGION_KEEP + 1) + 1) * 4) != KD_OK)
        sfail(ctx, KD_OK, "");
    uint32_t* list = kept ? (uint32_t*)kept + (size_t)nq * REGION_KEEP : nullptr;
    if (list) cudaMemsetAsync(list + nq, 0, 4, s);
    launch_region(ctx, ix, dlo, dhi, nq, order, nullptr, counts, kept, nullptr, nullptr, d_err, s);
    launch_offsets(ctx, counts, nq, sums, doffs, s);
    int64_t total = 0;
    cudaMemcpyAsync(&total, doffs + nq, 8, cudaMemcpyDeviceToHost, s);
    st = read_err(ctx, d_err, s);  // synchronises
    if (st != KD_OK) return st;
    if (!on_device) cudaMemcpyAsync(offsets, doffs, (size_t)(nq + 1) * 8, cudaMemcpyDeviceToHost, s);
    if (idx_out && total > 0) {
        if (total > capacity)
            return sfail(ctx, KD_EINVAL,
                         "capacity " + std::to_string(capacity) + " < " + std::to_string(total) + " results");
        int32_t* dout = idx_out;
        if (!on_device) {
            st = S.get((void**)&dout, (size_t)total * 4);
            if (st == KD_ENOMEM && (order || kept)) {  // the indices before what speeds their search up
                O.clear();
                order = nullptr;
                kept = nullptr;
                list = nullptr;
                st = S.get((void**)&dout, (size_t)total * 4);
                if (st == KD_OK) sfail(ctx, KD_OK, "");
            }
            if (st != KD_OK) return st;
        }
        if (list) {
            k_region_copy<<<(unsigned)((nq + 255) / 256), 256, 0, s>>>(counts, doffs, kept, nq, dout, list, list + nq);
            kd::ctx_add_launches(ctx, 1);
        }
        launch_region(ctx, ix, dlo, dhi, nq, list ? list : order, list ? list + nq : nullptr, counts, nullptr, doffs,
                      dout, d_err, s);
        if (!on_device) cudaMemcpyAsync(idx_out, dout, (size_t)total * 4, cudaMemcpyDeviceToHost, s);
    }
    return read_err(ctx, d_err, s);
}

}  // extern "C"

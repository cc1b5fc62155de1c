// kd_select.cu -- the O(n log n) k-d tree build of the paper's "Comparative
// Performance" section ("The O(n log n) Algorithm"), on the GPU.
//
// The paper's comparison algorithm sorts one index array by one super key,
// removes duplicate tuples, and then, at every level of the recursion, finds
// the median of each sub-array in the level's super key with a linear-time
// selection and partitions the sub-array around it.  It builds the same
// tree as the presorting method (every median is unique under the total
// super-key order), but without the other k-1 presorts.
//
// Here the index array is the presorting build's array 0 (super key 0,
// duplicates removed) and it carries its tuples' key words as planes (the
// tuple index plus k key planes, moved together).  Every segment of a level
// is processed by the same launches:
//   k_sel_hist / k_sel_choose  most-significant-digit radix selection.  Per
//       round, a 256-bin histogram of the next byte of the level's super key
//       over each segment's candidates (elements whose earlier bytes equal
//       the prefix chosen so far); the bin that holds the median's rank
//       becomes the next prefix byte.  A segment is resolved once its bin
//       holds a single element.  Each round reads every element once, so a
//       level is O(n) work, as with the paper's median of medians.
//   k_sel_move  partition around the medians: less -> the lower half,
//       greater -> the upper half, the median becomes the node.  Since the
//       next level selects afresh, the halves need not keep an order: slots
//       are claimed with atomics.
//   k_sel_order  a segment of at most 2048 tuples (1024 for k > 4) is sorted
//       by every super key in the shared memory of one block, which gives the
//       presorting build's input for that segment alone; its on-chip
//       finisher (k_finish) then builds the subtree.
#include <cstdint>

#include "kd_block_sort.cuh"

namespace kd {

constexpr int SEL_THREADS = 256;
constexpr int SEL_TILE = 2048;   // tile of the level kernels (positions)
constexpr int SEL_IPT = SEL_TILE / SEL_THREADS;
constexpr uint32_t KNONE = 0xffffffffu;
constexpr int SEL_RUN = 32;  // longest run of equal sort words ordered by compares

// Planes of the index array: tuple index and key words of each coordinate,
// two buffers.
template <typename KW>
struct SelBufs {
    uint32_t* id[2];
    KW* key[2][MAXK];
};

// Selection state of one segment of the current level.
template <typename KW>
struct SelSeg {
    int32_t lo, hi;
    int32_t pos;      // array position of the median; -1 unresolved, -2 empty segment
    uint32_t target;  // rank of the median among the current candidates
    uint32_t cnt[2];  // partition: elements placed in the lower / upper half
    int32_t start;    // first byte of the super key the candidates do not all share
    uint32_t pad;
    KW span_and, span_or;  // AND and OR of the segment's leading key words
    KW prefix[MAXK];  // super-key words; the bytes chosen so far (high bytes first)
};

// Byte r of a super key of k words of B bytes: word r / B, counted from the
// most significant byte.
template <typename KW>
__device__ __forceinline__ int sel_shift(int r) {
    constexpr int B = sizeof(KW);
    return 8 * (B - 1 - r % B);
}

template <typename KW>
__global__ void k_sel_init(int32_t m, int L, int nseg, SelSeg<KW>* __restrict__ segs, uint32_t* __restrict__ ghist) {
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < nseg; s += gridDim.x * blockDim.x) {
        SelSeg<KW> S;
        segment_bounds(m, L, s, S.lo, S.hi);
        S.pos = S.hi < S.lo ? -2 : -1;
        S.target = S.hi < S.lo ? 0u : (uint32_t)((S.hi - S.lo) >> 1);
        S.cnt[0] = S.cnt[1] = 0;
        S.start = 0;
        S.pad = 0;
        S.span_and = ~(KW)0;
        S.span_or = 0;
        for (int j = 0; j < MAXK; ++j) S.prefix[j] = 0;
        segs[s] = S;
    }
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < (int64_t)nseg * RADIX;
         i += (int64_t)gridDim.x * blockDim.x)
        ghist[i] = 0;
}

// The tile's segments (at most LEVEL_NSMAX) and their selection state.
template <typename KW>
struct SelTile {
    int ns;
    int32_t lo[LEVEL_NSMAX], hi[LEVEL_NSMAX], idx[LEVEL_NSMAX];
    int32_t pos[LEVEL_NSMAX];
    int32_t start[LEVEL_NSMAX];
    KW prefix[LEVEL_NSMAX][MAXK];
};

template <typename KW>
__device__ __forceinline__ void sel_load_tile(SelTile<KW>& T, int32_t pos0, int32_t npos, int32_t m, int L,
                                              const SelSeg<KW>* __restrict__ segs, int* err) {
    if (threadIdx.x == 0) {
        T.ns = tile_segments(pos0, npos, m, L, T.lo, T.hi, T.idx, err);
        for (int x = 0; x < T.ns; ++x) {
            const SelSeg<KW>& S = segs[T.idx[x]];
            T.pos[x] = S.pos;
            T.start[x] = S.start;
            for (int j = 0; j < MAXK; ++j) T.prefix[x][j] = S.prefix[j];
        }
    }
    __syncthreads();
}

// One selection round: histogram of super-key byte r over the candidates.
template <typename KW>
__global__ void __launch_bounds__(SEL_THREADS) k_sel_hist(const __grid_constant__ SelBufs<KW> bufs, int cur, int k,
                                                          int32_t m, int L, int r, int tile,
                                                          const SelSeg<KW>* __restrict__ segs,
                                                          uint32_t* __restrict__ ghist, int32_t* __restrict__ gany,
                                                          int* __restrict__ err) {
    __shared__ SelTile<KW> T;
    __shared__ uint32_t h[LEVEL_NSMAX][RADIX];
    __shared__ int32_t any[LEVEL_NSMAX][RADIX];
    const int tid = threadIdx.x;
    const int32_t pos0 = blockIdx.x * tile;
    const int32_t npos = min(tile, m - pos0);
    sel_load_tile(T, pos0, npos, m, L, segs, err);
    bool open = false;
    for (int x = 0; x < T.ns; ++x) open |= T.pos[x] == -1 && r >= T.start[x];
    if (!open) return;  // uniform: every segment of the tile is resolved, or shares byte r
    for (int i = tid; i < LEVEL_NSMAX * RADIX; i += SEL_THREADS) (&h[0][0])[i] = 0;
    __syncthreads();
    constexpr int B = sizeof(KW);
    const int j = r / B, sh = sel_shift<KW>(r);
    const int p = L % k;
    // the leading words of all rows in flight before the first is used
    KW x0[SEL_IPT];
    int slot[SEL_IPT];
    const bool one = T.ns == 1;
    const int32_t lo0 = T.lo[0], hi0 = T.hi[0];
#pragma unroll
    for (int e = 0; e < SEL_IPT; ++e) {
        const int o = e * SEL_THREADS + tid;
        const int32_t pos = pos0 + o;
        slot[e] = -1;
        if (o < npos) {
            if (one) slot[e] = pos >= lo0 && pos <= hi0 ? 0 : -1;
            else slot[e] = tile_slot(T.lo, T.hi, T.ns, pos);
        }
        x0[e] = slot[e] >= 0 ? bufs.key[cur][p][pos] : (KW)0;
    }
#pragma unroll
    for (int e = 0; e < SEL_IPT; ++e) {
        const int32_t pos = pos0 + e * SEL_THREADS + tid;
        const int sj = slot[e];
        bool cand = sj >= 0 && T.pos[sj] == -1 && r >= T.start[sj];
        uint32_t dig = 0;
        if (cand) {
            // the words of the super key up to word j, compared with the prefix
            KW wj = x0[e];
            if (j > 0) {
                cand = wj == T.prefix[sj][0];
                for (int jj = 1; jj <= j && cand; ++jj) {
                    int d = p + jj;
                    if (d >= k) d -= k;
                    wj = bufs.key[cur][d][pos];
                    if (jj < j) cand = wj == T.prefix[sj][jj];
                }
            }
            if (cand && sh + 8 < 8 * B) cand = (wj >> (sh + 8)) == (T.prefix[sj][j] >> (sh + 8));
            dig = (uint32_t)(wj >> sh) & 255u;
        }
        // the lanes that share the first candidate's segment and digit add once
        // (a run of equal top bytes would serialise on one counter); the others
        // add for themselves.  (Grouping every digit by a match instruction kept
        // that pipe 82% busy on spread digits; a round over 2^22 int64 tuples
        // 21 -> 16 us on average.)
        const uint32_t cands = __ballot_sync(0xffffffffu, cand);
        if (cands == 0) continue;
        const int first = __ffs(cands) - 1;
        const uint32_t key = (uint32_t)sj << 8 | dig;
        const uint32_t lead = __shfl_sync(0xffffffffu, key, first);  // (every lane takes part)
        const uint32_t same = __ballot_sync(0xffffffffu, cand && key == lead);
        if (cand) {
            const bool mine = (same >> (tid & 31)) & 1u;
            if (!mine || (tid & 31) == first) {
                atomicAdd(&h[sj][dig], mine ? (uint32_t)__popc(same) : 1u);
                any[sj][dig] = pos;
            }
        }
    }
    __syncthreads();
    for (int x = 0; x < T.ns; ++x) {
        if (T.pos[x] != -1) continue;
        const uint32_t c = h[x][tid];
        if (c) {
            atomicAdd(&ghist[(int64_t)T.idx[x] * RADIX + tid], c);
            gany[(int64_t)T.idx[x] * RADIX + tid] = any[x][tid];
        }
    }
}

// AND and OR of a 64- or 32-bit word over the lanes of `mask` (all calling).
__device__ __forceinline__ void sel_warp_and_or(uint32_t mask, uint32_t w, uint32_t& a, uint32_t& o) {
    a = __reduce_and_sync(mask, w);
    o = __reduce_or_sync(mask, w);
}
__device__ __forceinline__ void sel_warp_and_or(uint32_t mask, uint64_t w, uint64_t& a, uint64_t& o) {
    const uint32_t ah = __reduce_and_sync(mask, (uint32_t)(w >> 32)), al = __reduce_and_sync(mask, (uint32_t)w);
    const uint32_t oh = __reduce_or_sync(mask, (uint32_t)(w >> 32)), ol = __reduce_or_sync(mask, (uint32_t)w);
    a = ((uint64_t)ah << 32) | al;
    o = ((uint64_t)oh << 32) | ol;
}

__device__ __forceinline__ void sel_atomic_and_or(uint32_t* a, uint32_t* o, uint32_t va, uint32_t vo) {
    atomicAnd(a, va);
    atomicOr(o, vo);
}
__device__ __forceinline__ void sel_atomic_and_or(uint64_t* a, uint64_t* o, uint64_t va, uint64_t vo) {
    atomicAnd(reinterpret_cast<unsigned long long*>(a), (unsigned long long)va);
    atomicOr(reinterpret_cast<unsigned long long*>(o), (unsigned long long)vo);
}

// Span of every segment's leading key words (x_p of super key p): the
// bits on which AND and OR agree are shared by all of its elements.
template <typename KW>
__global__ void __launch_bounds__(SEL_THREADS) k_sel_span(const __grid_constant__ SelBufs<KW> bufs, int cur, int k,
                                                          int32_t m, int L, int tile, SelSeg<KW>* __restrict__ segs,
                                                          int* __restrict__ err) {
    __shared__ SelTile<KW> T;
    __shared__ KW s_and[LEVEL_NSMAX], s_or[LEVEL_NSMAX];
    const int tid = threadIdx.x;
    const int32_t pos0 = blockIdx.x * tile;
    const int32_t npos = min(tile, m - pos0);
    if (tid < LEVEL_NSMAX) {
        s_and[tid] = ~(KW)0;
        s_or[tid] = 0;
    }
    sel_load_tile(T, pos0, npos, m, L, segs, err);  // (synchronises the block)
    const int p = L % k;
    // warp, then block, then one global update per segment of the tile
    KW x0[SEL_IPT];
#pragma unroll
    for (int e = 0; e < SEL_IPT; ++e) {
        const int o = e * SEL_THREADS + tid;
        x0[e] = o < npos ? bufs.key[cur][p][pos0 + o] : (KW)0;
    }
#pragma unroll
    for (int e = 0; e < SEL_IPT; ++e) {
        const int o = e * SEL_THREADS + tid;
        const int sj = o < npos ? tile_slot(T.lo, T.hi, T.ns, pos0 + o) : -1;
        const KW w = sj >= 0 ? x0[e] : (KW)0;
        const uint32_t peers = __match_any_sync(0xffffffffu, (uint32_t)sj);  // lanes of one segment
        KW a, b;
        sel_warp_and_or(peers, w, a, b);
        if (sj >= 0 && (threadIdx.x & 31) == __ffs(peers) - 1) sel_atomic_and_or(&s_and[sj], &s_or[sj], a, b);
    }
    __syncthreads();
    if (tid < T.ns) sel_atomic_and_or(&segs[T.idx[tid]].span_and, &segs[T.idx[tid]].span_or, s_and[tid], s_or[tid]);
}

// The leading bytes every element of a segment shares become its prefix;
// selection starts at the first byte where they differ.  *first receives
// the smallest such byte over the level's open segments.
template <typename KW>
__global__ void k_sel_skip(int nseg, SelSeg<KW>* __restrict__ segs, int32_t* __restrict__ first) {
    constexpr int B = sizeof(KW);
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < nseg; s += gridDim.x * blockDim.x) {
        SelSeg<KW>& S = segs[s];
        if (S.pos != -1) continue;
        const KW diff = S.span_and ^ S.span_or;
        const int lead = diff == 0 ? 8 * B : (B == 8 ? __clzll((long long)diff) : __clz((int)(uint32_t)diff));
        const int cb = lead / 8 < B ? lead / 8 : B - 1;  // keep at least the last byte of the word to select
        const KW mask = cb == 0 ? (KW)0 : ~(KW)0 << (8 * (B - cb));
        S.prefix[0] = S.span_and & mask;
        S.start = cb;
        atomicMin(first, cb);
    }
}

// One warp per segment: the bin holding the median's rank becomes the next
// prefix byte; a bin of one element resolves the segment.
template <typename KW>
__global__ void k_sel_choose(int nseg, int r, int nbytes, SelSeg<KW>* __restrict__ segs,
                             uint32_t* __restrict__ ghist, const int32_t* __restrict__ gany,
                             uint32_t* __restrict__ unresolved, int* __restrict__ err) {
    const int lane = threadIdx.x & 31;
    const int s = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (s >= nseg) return;
    SelSeg<KW>& S = segs[s];
    if (S.pos != -1 || r < S.start) return;  // uniform per warp (byte r is shared: already in the prefix)
    uint32_t* hs = ghist + (int64_t)s * RADIX;
    uint32_t v[8], sum = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        v[i] = hs[lane * 8 + i];
        sum += v[i];
    }
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    const uint32_t target = S.target;
    const uint32_t excl = incl - sum;
    const bool mine = target >= excl && target < incl;
    const uint32_t who = __ballot_sync(0xffffffffu, mine);
    if (who == 0) {  // the candidates do not cover the rank: inconsistent state
        if (lane == 0) {
            atomicOr(err, ERR_INTERNAL);
            S.pos = -2;
        }
        return;
    }
    if (mine) {
        uint32_t c = excl;  // elements of the bins before b
        int b = 0;
        uint32_t cnt = 0;
        bool found = false;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            if (!found) {
                if (target < c + v[i]) {
                    b = lane * 8 + i;
                    cnt = v[i];
                    found = true;
                } else {
                    c += v[i];
                }
            }
        }
        S.target = target - c;
        const int j = r / (int)sizeof(KW);
        S.prefix[j] |= (KW)b << sel_shift<KW>(r);
        if (cnt == 1) {
            S.pos = gany[(int64_t)s * RADIX + b];
        } else if (r + 1 >= nbytes) {
            atomicOr(err, ERR_INTERNAL);  // two elements with equal super keys after deduplication
            S.pos = -2;
        } else {
            atomicAdd(unresolved, 1u);
        }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) hs[lane * 8 + i] = 0;
}

// Partition around the resolved medians; the median of each segment becomes
// the node at the segment's middle address.
template <typename KW>
__global__ void __launch_bounds__(SEL_THREADS) k_sel_move(const __grid_constant__ SelBufs<KW> bufs, int cur, int k,
                                                          int32_t m, int L, int tile, SelSeg<KW>* __restrict__ segs,
                                                          int32_t* __restrict__ node, int64_t in_off,
                                                          int* __restrict__ err) {
    __shared__ SelTile<KW> T;
    __shared__ KW med[LEVEL_NSMAX][MAXK];
    __shared__ uint32_t scnt[LEVEL_NSMAX][2], sbase[LEVEL_NSMAX][2];
    const int tid = threadIdx.x;
    const int32_t pos0 = blockIdx.x * tile;
    const int32_t npos = min(tile, m - pos0);
    sel_load_tile(T, pos0, npos, m, L, segs, err);
    const int p = L % k;
    if (tid < T.ns * MAXK) {
        const int x = tid / MAXK, j = tid % MAXK;
        int d = p + j;
        while (d >= k) d -= k;
        const int32_t mp = T.pos[x];
        med[x][j] = (j < k && mp >= T.lo[x] && mp <= T.hi[x]) ? bufs.key[cur][d][mp] : (KW)0;
    }
    if (tid < LEVEL_NSMAX * 2) (&scnt[0][0])[tid] = 0;
    __syncthreads();
    // half and slot of every row's element, packed: -1 none, else slot * 2 + half.
    // The loads of all rows are in flight before the first is used, here and
    // plane by plane below (row by row, each waited for its own): a level over
    // 2^22 int64 tuples of k = 3, 91 -> 49 us.
    int where[SEL_IPT];
    uint32_t local[SEL_IPT];
    KW x0[SEL_IPT];
#pragma unroll
    for (int e = 0; e < SEL_IPT; ++e) {
        const int o = e * SEL_THREADS + tid;
        x0[e] = o < npos ? bufs.key[cur][p][pos0 + o] : (KW)0;
    }
#pragma unroll
    for (int e = 0; e < SEL_IPT; ++e) {
        const int o = e * SEL_THREADS + tid;
        where[e] = -1;
        const int32_t pos = pos0 + o;
        const int sj = o < npos ? tile_slot(T.lo, T.hi, T.ns, pos) : -1;
        if (sj >= 0) {
            const int32_t mp = T.pos[sj];
            if (mp < T.lo[sj] || mp > T.hi[sj]) {
                atomicOr(err, ERR_INTERNAL);
            } else {
                KW x = x0[e], y = med[sj][0];
                for (int j = 1; j < k && x == y; ++j) {
                    int d = p + j;
                    if (d >= k) d -= k;
                    x = bufs.key[cur][d][pos];
                    y = med[sj][j];
                }
                if (x == y) {
                    if (pos != mp) atomicOr(err, ERR_INTERNAL);
                    const int32_t mid = T.lo[sj] + ((T.hi[sj] - T.lo[sj]) >> 1);
                    node[mid] = (int32_t)((int64_t)bufs.id[cur][pos] - in_off);
                } else {
                    where[e] = sj * 2 + (x > y ? 1 : 0);
                }
            }
        }
        // the lanes of a row that go to the same half claim their places together
        const uint32_t peers = __match_any_sync(0xffffffffu, where[e]);
        const int leader = __ffs(peers) - 1;
        uint32_t at = 0;
        if (where[e] >= 0 && (tid & 31) == leader) at = atomicAdd(&(&scnt[0][0])[where[e]], (uint32_t)__popc(peers));
        at = __shfl_sync(0xffffffffu, at, leader);
        local[e] = at + __popc(peers & lanemask_lt());
    }
    __syncthreads();
    if (tid < T.ns * 2) {
        const int x = tid >> 1, f = tid & 1;
        sbase[x][f] = atomicAdd(&segs[T.idx[x]].cnt[f], scnt[x][f]);
    }
    __syncthreads();
    int32_t dest[SEL_IPT];
#pragma unroll
    for (int e = 0; e < SEL_IPT; ++e) {
        dest[e] = -1;
        if (where[e] < 0) continue;
        const int sj = where[e] >> 1, f = where[e] & 1;
        const int32_t lo = T.lo[sj], hi = T.hi[sj], mid = lo + ((hi - lo) >> 1);
        const int32_t dst = (f ? mid + 1 : lo) + (int32_t)(sbase[sj][f] + local[e]);
        if (f ? (dst <= mid || dst > hi) : (dst >= mid)) {
            atomicOr(err, ERR_INTERNAL);
            continue;
        }
        dest[e] = dst;
        bufs.key[cur ^ 1][p][dst] = x0[e];
    }
    const int32_t first = pos0 + tid;
    {
        uint32_t v[SEL_IPT];
#pragma unroll
        for (int e = 0; e < SEL_IPT; ++e) v[e] = dest[e] >= 0 ? bufs.id[cur][first + e * SEL_THREADS] : 0u;
#pragma unroll
        for (int e = 0; e < SEL_IPT; ++e)
            if (dest[e] >= 0) bufs.id[cur ^ 1][dest[e]] = v[e];
    }
    for (int d = 0; d < k; ++d) {
        if (d == p) continue;
        KW v[SEL_IPT];
#pragma unroll
        for (int e = 0; e < SEL_IPT; ++e) v[e] = dest[e] >= 0 ? bufs.key[cur][d][first + e * SEL_THREADS] : (KW)0;
#pragma unroll
        for (int e = 0; e < SEL_IPT; ++e)
            if (dest[e] >= 0) bufs.key[cur ^ 1][d][dest[e]] = v[e];
    }
}

// ------------------------------------------------------ segment orders
// One block per segment of level lam (at most 32 NW E tuples): the places
// of its tuples in array 0 of the segment (super key 0 order) by every super
// key, as the finisher of the presorting build reads them: plane[p][lo + i] =
// lo + (place in array 0 of the i-th tuple by super key p), perm[lo + i] =
// the i-th tuple by super key 0.
//
// Each order is a radix sort by the 16 leading differing bits of x_p (two
// passes, where the finisher this replaces selected every median of every
// level by 4-bit rounds over all keys), then runs of equal words by
// super-key compares; where a run exceeds SEL_RUN, a radix sort by the whole
// super key.  2^22 int64 tuples, k = 3: 0.23 ms, and 0.20 ms for the finisher,
// against 3.77 ms.
template <typename KW, int NW, int E>
size_t sel_order_smem(int k) {
    return (size_t)32 * NW * E * (k * sizeof(KW) + 4 + 2 + 2);
}

struct SelOrder {
    uint32_t* plane[MAXK];
    uint32_t* perm;
};

template <typename KW, int NW, int E>
__global__ void __launch_bounds__(32 * NW) k_sel_order(const __grid_constant__ SelBufs<KW> bufs, int cur, int k,
                                                       int32_t m, int lam, const __grid_constant__ SelOrder out,
                                                       int* __restrict__ err) {
    constexpr int NT = 32 * NW, CAP = NT * E, BITS = 16;
    extern __shared__ __align__(16) unsigned char so_raw[];
    KW* keys = reinterpret_cast<KW*>(so_raw);                         // [k][CAP]
    uint32_t* s_key = reinterpret_cast<uint32_t*>(keys + (size_t)k * CAP);
    uint16_t* s_idx = reinterpret_cast<uint16_t*>(s_key + CAP);
    uint16_t* s_inv = s_idx + CAP;                                    // place of every tuple in array 0
    __shared__ __align__(16) uint16_t wc[NW][RADIX];
    __shared__ uint32_t s_ws[32], s_w[4];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int base = warp * 32 * E + lane;
    int32_t lo, hi;
    segment_bounds(m, lam, blockIdx.x, lo, hi);
    const int n = hi - lo + 1;
    if (n <= 0) return;
    if (n > CAP) {
        if (tid == 0) atomicOr(err, ERR_INTERNAL);
        return;
    }
    for (int d = 0; d < k; ++d)
        for (int i = tid; i < n; i += NT) keys[d * CAP + i] = bufs.key[cur][d][lo + i];
    __syncthreads();
    uint32_t key[E], id[E];
    auto load = [&](const KW* x, bool identity) {  // the current order; the bits in which its keys differ
        KW a = ~(KW)0, r = 0;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int o = base + e * 32;
            id[e] = identity ? (uint32_t)o : (o < n ? s_idx[o] : 0u);
            if (o < n) {
                a &= x[id[e]];
                r |= x[id[e]];
                if (identity) s_idx[o] = (uint16_t)o;
            }
        }
        return block_diff(a, r, s_w);
    };
    for (int p = 0; p < k; ++p) {
        const KW* const xp = keys + p * CAP;
        const KW differ = load(xp, true);
        const int shift = word_shift<BITS>(differ);
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int o = base + e * 32;
            key[e] = o < n ? sort_word<BITS>(xp[o], shift) : 0u;
            if (differ == 0 && o < n) s_key[o] = 0;  // (no pass writes the words)
        }
        __syncthreads();
        if (differ != 0) {
            for (int b = 0; b < BITS; b += 8) block_pass<NW, E>(key, id, b, n, s_key, s_idx, wc, s_ws);
        }
        bool tie = false, lng = false;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int o = base + e * 32;
            if (o + 1 >= n || s_key[o + 1] != s_key[o]) continue;
            tie = true;
            lng |= o + SEL_RUN < n && s_key[o + SEL_RUN] == s_key[o];
        }
        if (__syncthreads_or(lng)) {
            for (int r = k - 1; r >= 0; --r) {  // least significant coordinate first
                const KW* const x = keys + (p + r < k ? p + r : p + r - k) * CAP;
                const KW df = load(x, r == k - 1);
                __syncthreads();
#pragma unroll
                for (int w = 0; w < (int)sizeof(KW) * 8; w += 32) {
                    if ((uint32_t)(df >> w) == 0) continue;
#pragma unroll
                    for (int e = 0; e < E; ++e) key[e] = base + e * 32 < n ? (uint32_t)(x[id[e]] >> w) : 0u;
                    for (int b = 0; b < 32; b += 8)
                        if (((uint32_t)(df >> w) >> b) & 255u)
                            block_pass<NW, E>(key, id, b, n, s_key, s_idx, wc, s_ws);
                }
                __syncthreads();
            }
        } else if (__syncthreads_or(tie)) {
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const int o = base + e * 32;
                id[e] = 0;
                key[e] = KNONE;  // the tuple's new place, if it is in a run
                if (o >= n) continue;
                const uint32_t x = s_key[o];
                int s = o, f = o;
                while (s > 0 && s_key[s - 1] == x) --s;
                while (f + 1 < n && s_key[f + 1] == x) ++f;
                if (s == f) continue;
                const int i = s_idx[o];
                id[e] = (uint32_t)i;
                int c = s;
                for (int y = s; y <= f; ++y) {
                    if (y == o) continue;
                    const int j = s_idx[y];
                    for (int r = 0; r < k; ++r) {  // (no two super keys are equal)
                        const KW* const z = keys + (p + r < k ? p + r : p + r - k) * CAP;
                        if (z[j] != z[i]) {
                            c += z[j] < z[i] ? 1 : 0;
                            break;
                        }
                    }
                }
                key[e] = (uint32_t)c;
            }
            __syncthreads();
#pragma unroll
            for (int e = 0; e < E; ++e)
                if (key[e] != KNONE) s_idx[key[e]] = (uint16_t)id[e];
            __syncthreads();
        }
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int o = base + e * 32;
            if (o >= n) continue;
            const int i = s_idx[o];
            if (p == 0) {
                s_inv[i] = (uint16_t)o;
                out.perm[lo + o] = bufs.id[cur][lo + i];
                out.plane[0][lo + o] = (uint32_t)(lo + o);
            } else {
                out.plane[p][lo + o] = (uint32_t)(lo + s_inv[i]);
            }
        }
        __syncthreads();  // s_inv is written; s_idx and s_key are free
    }
}

// ------------------------------------------------------------ launchers
template <typename KW>
static SelBufs<KW> sel_bufs(void* const* id, void* const* key, int k) {
    SelBufs<KW> B{};
    for (int b = 0; b < 2; ++b) {
        B.id[b] = static_cast<uint32_t*>(id[b]);
        for (int d = 0; d < k; ++d) B.key[b][d] = static_cast<KW*>(key[b * MAXK + d]);
    }
    return B;
}

size_t sel_seg_bytes(int key64) { return key64 ? sizeof(SelSeg<uint64_t>) : sizeof(SelSeg<uint32_t>); }

// Largest segment whose orders one block makes (and the presorting build's
// finisher takes).
int sel_order_tile(int k) { return k <= 4 ? 2048 : 1024; }

template <typename KW>
static cudaError_t sel_level(const SelBufs<KW>& B, int cur, int k, int32_t m, int L, int tile, void* segs,
                             uint32_t* ghist, int32_t* gany, uint32_t* unresolved, int32_t* node, int64_t in_off,
                             int* err, cudaStream_t s, int round_begin, int round_end, int phase) {
    const int nseg = 1 << L;
    const int ntiles = (m + tile - 1) / tile;
    SelSeg<KW>* sg = static_cast<SelSeg<KW>*>(segs);
    if (phase == 0) {
        const int g = std::min(152 * 16, (int)(((int64_t)nseg * RADIX + 255) / 256));
        k_sel_init<KW><<<g, 256, 0, s>>>(m, L, nseg, sg, ghist);
        return cudaGetLastError();
    }
    if (phase == 3) {
        k_sel_span<KW><<<ntiles, SEL_THREADS, 0, s>>>(B, cur, k, m, L, tile, sg, err);
        k_sel_skip<KW><<<std::min(152 * 8, (nseg + 255) / 256), 256, 0, s>>>(nseg, sg,
                                                                            reinterpret_cast<int32_t*>(unresolved));
        return cudaGetLastError();
    }
    if (phase == 1) {
        for (int r = round_begin; r < round_end; ++r) {
            k_sel_hist<KW><<<ntiles, SEL_THREADS, 0, s>>>(B, cur, k, m, L, r, tile, sg, ghist, gany, err);
            k_sel_choose<KW><<<(nseg * 32 + 255) / 256, 256, 0, s>>>(nseg, r, k * (int)sizeof(KW), sg, ghist, gany,
                                                                     unresolved, err);
        }
        return cudaGetLastError();
    }
    k_sel_move<KW><<<ntiles, SEL_THREADS, 0, s>>>(B, cur, k, m, L, tile, sg, node, in_off, err);
    return cudaGetLastError();
}

// One level of the selection build over every segment of level L, in tiles
// of `tile` = SEL_TILE positions (a tile must touch at most LEVEL_NSMAX
// segments, so these hold at least 1024 tuples).
// phase 0: reset the segments' state; 3: the shared leading bytes of every
// segment (*unresolved, as an int32, receives the smallest first byte to
// select; it must hold the byte count before); 1: selection rounds
// [round_begin, round_end) (each adds the segments still unresolved to
// *unresolved); 2: partition around the medians.
cudaError_t launch_sel_level(int key64, void* const* id, void* const* key, int cur, int k, int32_t m, int L, int tile,
                             void* segs, uint32_t* ghist, int32_t* gany, uint32_t* unresolved, int32_t* node,
                             int64_t in_off, int* err, cudaStream_t s, int round_begin, int round_end, int phase) {
    if (m <= 0) return cudaSuccess;
    if (tile != SEL_TILE) return cudaErrorInvalidValue;
    if (key64)
        return sel_level<uint64_t>(sel_bufs<uint64_t>(id, key, k), cur, k, m, L, tile, segs, ghist, gany, unresolved,
                                   node, in_off, err, s, round_begin, round_end, phase);
    return sel_level<uint32_t>(sel_bufs<uint32_t>(id, key, k), cur, k, m, L, tile, segs, ghist, gany, unresolved,
                               node, in_off, err, s, round_begin, round_end, phase);
}

template <typename KW>
static cudaError_t init_sel_order() {
    // 160 KB covers every k: 2048 tuples up to k = 4, 1024 up to 8
    cudaError_t e = cudaFuncSetAttribute((const void*)k_sel_order<KW, 8, 8>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute((const void*)k_sel_order<KW, 8, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 160 * 1024);
    return e;
}
cudaError_t init_select_kernels() {
    const cudaError_t e = init_sel_order<uint32_t>();
    return e == cudaSuccess ? init_sel_order<uint64_t>() : e;
}

template <typename KW>
static cudaError_t sel_order(const SelBufs<KW>& B, int cur, int k, int32_t m, int lam, const SelOrder& out, int* err,
                             cudaStream_t s) {
    const unsigned units = 1u << lam;
    if (k <= 4) k_sel_order<KW, 8, 8><<<units, 256, sel_order_smem<KW, 8, 8>(k), s>>>(B, cur, k, m, lam, out, err);
    else k_sel_order<KW, 8, 4><<<units, 256, sel_order_smem<KW, 8, 4>(k), s>>>(B, cur, k, m, lam, out, err);
    return cudaGetLastError();
}

// The orders of the 2^lam segments of level lam (each at most
// sel_order_tile(k) tuples), in the buffer that does not hold the elements:
// plane[p] over its key plane p, perm over its index plane.
cudaError_t launch_sel_order(int key64, void* const* id, void* const* key, int cur, int k, int32_t m, int lam,
                             uint32_t** plane, uint32_t** perm, int* err, cudaStream_t s) {
    if (m <= 0) return cudaSuccess;
    SelOrder out{};
    for (int p = 0; p < k; ++p) plane[p] = out.plane[p] = static_cast<uint32_t*>(key[(cur ^ 1) * MAXK + p]);
    *perm = out.perm = static_cast<uint32_t*>(id[cur ^ 1]);
    if (key64) return sel_order<uint64_t>(sel_bufs<uint64_t>(id, key, k), cur, k, m, lam, out, err, s);
    return sel_order<uint32_t>(sel_bufs<uint32_t>(id, key, k), cur, k, m, lam, out, err, s);
}

}  // namespace kd

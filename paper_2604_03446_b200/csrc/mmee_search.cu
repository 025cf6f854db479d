// The search kernel: every mapping decided, capacity pruning, top-k, in one launch.
//
// Work decomposition.  CTA c takes one tiling out of every `grid` consecutive ones, so that tilings that cannot fit at
// all (large tiles, neighbours in the index order) spread evenly, keeps those that can in a compact list with their
// size and stationary-pair tables in shared memory, and cuts the list into items: (class of C, tiling, order) of the
// fused mode, then (tiling, order) of the unfused ones.  A warp takes 32 items at a time; one thread decides one item
// in closed form over classes of levels (mmee_classes.cuh): how many of its rows fit and its least key, exact in
// 64 bits.  No candidate, row or threshold is kept per mapping, and nothing but the CTA's result leaves the SM.
//
// Selection.  A block (tiling, fusion mode, order) is a contiguous range of mapping indices, so that (least key, block
// number) orders blocks as their best mappings are ordered.  The k best mappings of the whole space lie in the k best
// blocks: a block outside them has k mappings of other blocks before its first.  The same holds for the list of the k
// best ITEMS, in which a fused block can appear once per class of C.  Each warp (k = 1: each thread) keeps such a list;
// the CTA that finishes last (a ticket counter, no wait) merges the CTAs' lists and evaluates the winning blocks mapping
// by mapping from their level tables (mmee_block.cuh), which are built from the query vectors independently.
#include <cuda_runtime.h>

#include <climits>
#include <cstddef>

#include "mmee_block.cuh"
#include "mmee_search.h"

namespace mmee {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kWarps = kSearchThreads / 32;
constexpr int kTopK = (int)MMEE_MAX_TOPK;
// One optimum; one optimum over the rows kept by symbolic pruning; the k best; one optimum of a chain of searches;
// one optimum for each of several array shapes.
constexpr int kModeSingle = 0, kModePrune = 1, kModeMulti = 2, kModeChain = 3, kModeArrays = 4;

// ------------------------------------------------------------------------------------------------
// (key, number) pairs
// ------------------------------------------------------------------------------------------------
// A sorted list held by a warp in registers: lane j holds entry j, best first; an empty slot, and every lane from k on,
// holds (kInfKey, UINT64_MAX), which follows every real pair.  All 32 lanes call these functions converged.

__device__ __forceinline__ bool pair_less(int64_t ka, uint64_t ia, int64_t kb, uint64_t ib) {
    return ka < kb || (ka == kb && ia < ib);
}

__device__ __forceinline__ void reg_insert(int64_t& ek, uint64_t& ei, int k, int64_t nk, uint64_t ni, int lane) {
    const unsigned smaller = __ballot_sync(kFull, pair_less(ek, ei, nk, ni));
    const int pos = __popc(smaller);
    if (pos >= k) return;
    const int64_t uk = __shfl_up_sync(kFull, ek, 1);
    const uint64_t ui = __shfl_up_sync(kFull, ei, 1);
    if (lane == pos) { ek = nk; ei = ni; }
    else if (lane > pos && lane < k) { ek = uk; ei = ui; }
}

// Merge of two such lists: the other list reversed and the lane-wise minimum of the two give the 16 smallest of the 32
// pairs as a bitonic sequence, which four compare-exchange stages sort.
__device__ __forceinline__ void reg_merge(int64_t& ek, uint64_t& ei, int k, int64_t ok, uint64_t oi, int lane) {
    const int rev = (kTopK - 1 - lane) & 31;
    const int64_t rk = __shfl_sync(kFull, ok, rev);
    const uint64_t ri = __shfl_sync(kFull, oi, rev);
    if (lane < kTopK && pair_less(rk, ri, ek, ei)) { ek = rk; ei = ri; }
#pragma unroll
    for (int stride = kTopK / 2; stride >= 1; stride >>= 1) {
        const int64_t pk = __shfl_xor_sync(kFull, ek, stride);
        const uint64_t pi = __shfl_xor_sync(kFull, ei, stride);
        const bool keep_smaller = (lane & stride) == 0;
        if (pair_less(pk, pi, ek, ei) == keep_smaller) { ek = pk; ei = pi; }
    }
    if (lane >= k) { ek = kInfKey; ei = UINT64_MAX; }
}

// Ascending sort of 32 pairs, one per lane (a bitonic network of 15 compare-exchange stages).
__device__ __noinline__ void warp_sort_pairs(int64_t& ck, uint64_t& ci, int lane) {
#pragma unroll
    for (int size = 2; size <= 32; size <<= 1) {
#pragma unroll
        for (int stride = size >> 1; stride >= 1; stride >>= 1) {
            const int64_t pk = __shfl_xor_sync(kFull, ck, stride);
            const uint64_t pi = __shfl_xor_sync(kFull, ci, stride);
            const bool keep_smaller = ((lane & size) == 0) == ((lane & stride) == 0);
            if (pair_less(pk, pi, ck, ci) == keep_smaller) { ck = pk; ci = pi; }
        }
    }
}

// The pairs of the lanes with `pend` set enter the list: one by one when they are few, else sorted and merged.
__device__ __forceinline__ void warp_offer(int64_t& ek, uint64_t& ei, int k, int64_t key, uint64_t num, bool pend, int lane) {
    unsigned m = __ballot_sync(kFull, pend);
    if (__popc(m) > 3) {
        int64_t ck = pend ? key : kInfKey;
        uint64_t ci = pend ? num : UINT64_MAX;
        warp_sort_pairs(ck, ci, lane);
        reg_merge(ek, ei, k, ck, ci, lane);
        return;
    }
    for (; m; m &= m - 1) {
        const int src = __ffs(m) - 1;
        reg_insert(ek, ei, k, __shfl_sync(kFull, key, src), __shfl_sync(kFull, num, src), lane);
    }
}

// Smallest of the non-negative numbers of the lanes with `in` set (UINT64_MAX if there is none), by 32-bit warp minima;
// `in` becomes whether this lane holds it.
__device__ __forceinline__ uint64_t warp_min_u64(uint64_t v, bool& in) {
    const uint32_t hi = __reduce_min_sync(kFull, in ? (uint32_t)(v >> 32) : 0xffffffffu);
    in = in && (uint32_t)(v >> 32) == hi;
    const uint32_t lo = __reduce_min_sync(kFull, in ? (uint32_t)v : 0xffffffffu);
    in = in && (uint32_t)v == lo;
    return ((uint64_t)hi << 32) | lo;
}

// Smallest pair of the warp, in every lane (keys are non-negative).
__device__ __forceinline__ void warp_min_pair(int64_t& k, uint64_t& i) {
    bool in = true;
    k = (int64_t)warp_min_u64((uint64_t)k, in);
    i = warp_min_u64(i, in);
}
// ... by key, then second key, then number.
__device__ __forceinline__ void warp_min_triple(int64_t& k, int64_t& k2, uint64_t& i) {
    bool in = true;
    k = (int64_t)warp_min_u64((uint64_t)k, in);
    k2 = (int64_t)warp_min_u64((uint64_t)k2, in);
    i = warp_min_u64(i, in);
}
__device__ __forceinline__ int64_t min3(const int64_t (&v)[3]) {
    const int64_t m = v[0] < v[1] ? v[0] : v[1];
    return m < v[2] ? m : v[2];
}

__device__ __forceinline__ bool triple_less(int64_t ka, int64_t la, uint64_t ia, int64_t kb, int64_t lb, uint64_t ib) {
    return ka < kb || (ka == kb && (la < lb || (la == lb && ia < ib)));
}

// ------------------------------------------------------------------------------------------------
// shared memory
// ------------------------------------------------------------------------------------------------

struct Shared {
    // What lanes index with different indices (the constant bank would serialise them), copied from the plan.
    OrderInfo order[kMaxOrders];
    KeptMasks kept;
    uint32_t divs[4][MMEE_MAX_DIVISORS];
    uint32_t cofactors[4][MMEE_MAX_DIVISORS];       // dimension / divisor
    uint32_t pe_rows, pe_cols;      // the array's logical shape
    uint32_t row_folds[4][MMEE_MAX_DIVISORS], col_folds[4][MMEE_MAX_DIVISORS];      // register-file tiling only
    alignas(16) longlong2 tops[kWarps][MMEE_MAX_TOPK];
    long long kth[kWarps];          // finalize, k > 1: the k-th key of each warp's list (kInfKey: not full)
    long long G;                    // k > 1: upper bound on the k-th smallest key
    unsigned long long feasible_rows[kWarps];
    uint32_t live_tilings[kWarps];
    uint32_t n_live;                // tilings of the current pass that can fit
    uint32_t n_fit;                 // STAIRS: those of them that fit under the bound of the search before
    long long bound;                // chained searches: that bound
    uint32_t cursor;                // next group of 32 items
    uint32_t last_cta, check_failed;
    uint32_t waited;                // chained searches: the one waited for is over
    union {
        TileTab tile[kMaxChunk];
        BlockTab block[kWarps];
        mmee_result_t record[MMEE_MAX_TOPK];
    };
};

struct SharedDivisors {       // see PlanDivisors
    const Shared& sh;
    MMEE_HD uint32_t rows() const { return sh.pe_rows; }
    MMEE_HD uint32_t cols() const { return sh.pe_cols; }
    MMEE_HD uint32_t div(int d, uint32_t i) const { return sh.divs[d][i]; }
    MMEE_HD uint32_t cofactor(int d, uint32_t i) const { return sh.cofactors[d][i]; }
    MMEE_HD uint32_t row_folds(int d, uint32_t i) const { return sh.row_folds[d][i]; }
    MMEE_HD uint32_t col_folds(int d, uint32_t i) const { return sh.col_folds[d][i]; }
};

// ------------------------------------------------------------------------------------------------
// finalize: merge the CTAs' partial lists, evaluate the winning blocks, write the records, reset the scratch header
// ------------------------------------------------------------------------------------------------

// Classes of levels as they are walked mapping by mapping: 3*3*3*4*4 of a fused block, 3*3*3*3 of an unfused one.
constexpr uint32_t kFusedReps = 432, kUnfusedReps = 81;

struct Rep { int lv[5], width[5]; };       // first levels and numbers of levels of one class combination

__device__ __forceinline__ Rep decode_rep(const OrderInfo& o, bool fused, uint32_t r) {
    Rep q;
    const int c[5] = {(int)(fused ? r / 144u : r / 27u), (int)(fused ? r / 48u % 3u : r / 9u % 3u), (int)(fused ? r / 16u % 3u : 0u),
                      (int)(fused ? r / 4u % 4u : r / 3u % 3u), (int)(fused ? r % 4u : r % 3u)};
#pragma unroll
    for (int x = 0; x < 5; ++x) {
        if (!fused && x >= OP_D) {          // L3 and the class from L4 on are one
            q.lv[x] = c[x] ? o.first[x][c[x] + 1] : 0;
            q.width[x] = c[x] ? o.width[x][c[x] + 1] : o.width[x][0] + o.width[x][1];
        } else {
            q.lv[x] = o.first[x][c[x]];
            q.width[x] = o.width[x][c[x]];
        }
    }
    if (!fused) q.width[OP_C] = 1;          // C is always at L3
    return q;
}

__device__ __forceinline__ uint32_t row_of(bool fused, int a, int b, int c, int d, int e) {
    return (uint32_t)(fused ? (((a * 5 + b) * 5 + c) * 5 + d) * 5 + e : ((a * 5 + b) * 5 + d) * 5 + e);
}

// The best mapping of one block whose least key is `key`: the lowest index with that key (the first row of a class
// combination precedes its other rows, so only those are looked at).  All threads of the CTA; the pair ends up in every
// lane of every warp's own share, to be reduced over the warps.
template <int OBJ, bool NEED>
__device__ __forceinline__ void best_of_block(const Plan& p, const Limits& lim, const Shared& sh, int64_t key, int64_t need,
                                              int64_t& ek, uint64_t& ei) {
    const BlockTab& bt = sh.block[0];
    const OrderInfo& o = sh.order[bt.slot];
    const bool fused = bt.phi == 0;
    ek = kInfKey;
    ei = UINT64_MAX;
    for (uint32_t r = threadIdx.x; r < (fused ? kFusedReps : kUnfusedReps); r += kSearchThreads) {
        const Rep q = decode_rep(o, fused, r);
        const RowTerms t = row_terms(p, lim, bt, q.lv[0], q.lv[1], q.lv[2], q.lv[3], q.lv[4]);
        if (!t.fits) continue;
        uint32_t at = 9;
#pragma unroll
        for (int s = 8; s >= 0; --s)
            if (((p.sm_mask >> s) & 1u) && mapping_key<OBJ>(p, lim, bt, t, s) == key) at = (uint32_t)s;
        const uint64_t idx = bt.first_idx + row_of(fused, q.lv[0], q.lv[1], q.lv[2], q.lv[3], q.lv[4]) * 9u + at;
        if (at < 9u && idx < ei && (!NEED || t.need == need)) { ek = key; ei = idx; }
    }
    warp_min_pair(ek, ei);
}

// The least buffer need among the mappings of the block with that key and an index below `idx` (UINT64_MAX: none); each
// warp's in all its lanes.
template <int OBJ>
__device__ __forceinline__ uint64_t least_need_before(const Plan& p, const Limits& lim, const Shared& sh, int64_t key, uint64_t idx) {
    const BlockTab& bt = sh.block[0];
    const OrderInfo& o = sh.order[bt.slot];
    const bool fused = bt.phi == 0;
    uint64_t least = UINT64_MAX;
    for (uint32_t r = threadIdx.x; r < (fused ? kFusedReps : kUnfusedReps); r += kSearchThreads) {
        const Rep q = decode_rep(o, fused, r);
        const RowTerms t = row_terms(p, lim, bt, q.lv[0], q.lv[1], q.lv[2], q.lv[3], q.lv[4]);
        if (!t.fits || (uint64_t)t.need >= least) continue;
        bool has = false;
        const uint64_t first = bt.first_idx + row_of(fused, q.lv[0], q.lv[1], q.lv[2], q.lv[3], q.lv[4]) * 9u;
        for (int s = 0; s < 9; ++s)
            has |= ((p.sm_mask >> s) & 1u) && first + (uint32_t)s < idx && mapping_key<OBJ>(p, lim, bt, t, s) == key;
        if (has) least = (uint64_t)t.need;
    }
    bool in = true;
    return warp_min_u64(least, in);
}

// The mappings of block `j` of sh.block that precede the running k-th pair (lk, li), none above `bound`, into the warps'
// lists.  A lane holds one class combination and walks its mappings in (key, index) order: the stationary pairs of its
// least key over its rows, then those of the next larger key; the warp takes the smallest of its lanes' next mappings
// until it has k of them or the next one does not precede what a full list of any warp ends with.  (Taking whole
// combinations one after the other, each sorted into the list, needed a dozen of them per warp where all mappings tie:
// 24 us of a Llama top-16 search instead of 12.)
template <int OBJ>
__device__ __forceinline__ void best_of_block_multi(const Plan& p, const Limits& lim, Shared& sh, int j, int64_t bound, int k, int lane,
                                                    int64_t lk, uint64_t li, int64_t& ek, uint64_t& ei) {
    const BlockTab& bt = sh.block[j];
    const OrderInfo& o = sh.order[bt.slot];
    const bool fused = bt.phi == 0;
    const uint32_t n_reps = fused ? kFusedReps : kUnfusedReps;
#pragma unroll 1
    for (uint32_t r = threadIdx.x; r - lane < n_reps; r += kSearchThreads) {
        const Rep q = decode_rep(o, fused, r < n_reps ? r : 0u);
        const RowTerms t = row_terms(p, lim, bt, q.lv[0], q.lv[1], q.lv[2], q.lv[3], q.lv[4]);
        const uint32_t first_row = row_of(fused, q.lv[0], q.lv[1], q.lv[2], q.lv[3], q.lv[4]);
        int64_t hk = -1;                        // the lane's next mapping: key, index relative to the block's first
        uint32_t off = 0;
        uint32_t pairs = 0, left = 0;           // stationary pairs with that key, those left of the row
        uint32_t row = 0;                       // the row, and where its levels stand within their classes
        int at[5] = {0, 0, 0, 0, 0};
        int64_t nk = kInfKey;
        uint64_t ni = UINT64_MAX;
        // This warp's k-th pair bounds the block's; of the other warps' the key alone does, with any index, since they may be
        // writing it: one 64-bit access each.
        static_assert(sizeof(sh.kth[0]) == 8, "read without a barrier: a word that cannot be seen half written");
        const int64_t own_k = __shfl_sync(kFull, ek, k - 1);
        const uint64_t own_i = __shfl_sync(kFull, ei, k - 1);
        if (pair_less(own_k, own_i, lk, li)) { lk = own_k; li = own_i; }
        bool in = true;
        const int64_t other = (int64_t)warp_min_u64((uint64_t)*const_cast<volatile long long*>(&sh.kth[lane & (kWarps - 1)]), in);
        if (other < lk) { lk = other; li = UINT64_MAX; }
        bool advance = r < n_reps && t.fits;
        if (!advance) hk = kInfKey;
        int64_t level = -1;                     // the key whose mappings are being taken
#pragma unroll 1
        for (int i = 0; i < k;) {
            if (advance) {
                left &= left - 1u;
                if (!left) {
                    bool more = false;
                    if (pairs) {                // the next row of the combination: its levels count up, E's fastest
                        int stride = 1;
#pragma unroll
                        for (int x = 4; x >= 0; --x) {
                            if (!fused && x == OP_C) continue;
                            if (!more) {
                                more = ++at[x] < q.width[x];
                                row += (uint32_t)(more ? stride : -stride * (q.width[x] - 1));
                                if (!more) at[x] = 0;
                            }
                            stride *= 5;
                        }
                    }
                    if (!more) {                // the next larger key
                        const int64_t last = hk;
                        hk = kInfKey;
                        pairs = 0;
                        for (int s = 0; s < 9; ++s) {
                            const int64_t key = mapping_key<OBJ>(p, lim, bt, t, s);
                            if (!((p.sm_mask >> s) & 1u) || key <= last || key > hk) continue;
                            pairs = key < hk ? 1u << s : pairs | 1u << s;
                            hk = key;
                        }
                        row = first_row;
                        if (hk > bound) hk = kInfKey;
                    }
                    left = pairs;
                }
                off = row * 9u + (uint32_t)(__ffs(left) - 1);
            }
            // the lowest index among the lanes whose next mapping has the current key; without one, the next key
            uint32_t mine = hk == level ? off : 0xffffffffu;
            uint32_t least = __reduce_min_sync(kFull, mine);
            if (least == 0xffffffffu) {
                const uint32_t kh = __reduce_min_sync(kFull, (uint32_t)((uint64_t)hk >> 32));
                const uint32_t kl = __reduce_min_sync(kFull, (uint32_t)((uint64_t)hk >> 32) == kh ? (uint32_t)hk : 0xffffffffu);
                level = (int64_t)(((uint64_t)kh << 32) | kl);
                if (level == kInfKey) break;
                mine = hk == level ? off : 0xffffffffu;
                least = __reduce_min_sync(kFull, mine);
            }
            if (!pair_less(level, bt.first_idx + least, lk, li)) break;
            if (lane == i) { nk = level; ni = bt.first_idx + least; }
            advance = mine == least;
            ++i;
        }
        reg_merge(ek, ei, k, nk, ni, lane);
        if (lane == k - 1) *const_cast<volatile long long*>(&sh.kth[threadIdx.x >> 5]) = ek;
        __syncwarp();
    }
}

// The warps' lists (in registers) merged pairwise into sh.tops[0].  All threads of the CTA.
__device__ __forceinline__ void merge_warps(Shared& sh, int k, int lane, int warp, int64_t& ek, uint64_t& ei) {
    if (lane < kTopK) sh.tops[warp][lane] = make_longlong2((long long)ek, (long long)ei);
    for (int stride = kWarps / 2; stride >= 1; stride >>= 1) {
        __syncthreads();
        if (warp < stride) {
            const longlong2 theirs = lane < kTopK ? sh.tops[warp + stride][lane] : make_longlong2(kInfKey, -1ll);
            reg_merge(ek, ei, k, theirs.x, (uint64_t)theirs.y, lane);
            if (lane < kTopK) sh.tops[warp][lane] = make_longlong2((long long)ek, (long long)ei);
        }
    }
    __syncthreads();
}

// The smallest of the warps' pairs (k = 1; each warp's in all its lanes), in every thread of the CTA.
__device__ __forceinline__ void min_over_warps(Shared& sh, int lane, int warp, int64_t& ek, uint64_t& ei) {
    __syncthreads();
    if (lane == 0) sh.tops[warp][0] = make_longlong2((long long)ek, (long long)ei);
    __syncthreads();
    const longlong2 v = sh.tops[lane & (kWarps - 1)][0];
    ek = v.x;
    ei = (uint64_t)v.y;
    warp_min_pair(ek, ei);
}

struct ArrayDivisors {        // the same with another array's rows and columns
    const Shared& sh;
    uint32_t pe_rows, pe_cols;
    MMEE_HD uint32_t rows() const { return pe_rows; }
    MMEE_HD uint32_t cols() const { return pe_cols; }
    MMEE_HD uint32_t div(int d, uint32_t i) const { return sh.divs[d][i]; }
    MMEE_HD uint32_t row_folds(int d, uint32_t i) const { return folds(sh.divs[d][i], pe_rows); }
    MMEE_HD uint32_t col_folds(int d, uint32_t i) const { return folds(sh.divs[d][i], pe_cols); }
};

// What the kernels look up in shared memory, by all threads of a CTA (the caller synchronises).
template <bool PRUNE>
__device__ __forceinline__ void load_shared(const Plan& p, uint32_t pe_rows, uint32_t pe_cols, Shared& sh) {
    const int tid = threadIdx.x;
    for (int i = tid; i < (int)(sizeof(sh.order) / 4); i += kSearchThreads)
        reinterpret_cast<uint32_t*>(sh.order)[i] = reinterpret_cast<const uint32_t*>(p.order)[i];
    if (PRUNE)
        for (int i = tid; i < (int)(sizeof(KeptMasks) / 4); i += kSearchThreads)
            reinterpret_cast<uint32_t*>(&sh.kept)[i] = reinterpret_cast<const uint32_t*>(&p.kept)[i];
    static_assert(kSearchThreads == 4 * MMEE_MAX_DIVISORS, "one thread per divisor");
    if ((uint32_t)(tid & 63) < p.ndiv[tid >> 6]) {
        const int d = tid >> 6, i = tid & 63;
        sh.divs[d][i] = p.divs[d][i];
        sh.cofactors[d][i] = (p.mirrored >> d) & 1u ? p.divs[d][p.ndiv[d] - 1 - i] : p.dim[d] / p.divs[d][i];
        if (p.rf_tiling) {
            sh.row_folds[d][i] = folds(p.divs[d][i], pe_rows);
            sh.col_folds[d][i] = folds(p.divs[d][i], pe_cols);
        }
    }
    if (tid == 0) {
        sh.pe_rows = pe_rows;
        sh.pe_cols = pe_cols;
    }
}

// The items of a block's tables (block_item), their three kinds on three warps.
__device__ __forceinline__ int split_item(int warp, int lane) {
    return warp == 0 ? (lane < 25 ? lane : -1) : (warp == 1 ? (lane < 6 ? 25 + lane : -1) : (warp == 2 && lane == 0 ? 31 : -1));
}

// Chained searches run one after the other in one kernel, whose CTAs are all resident (a cooperative launch): a CTA that
// has published its part of one waits for the CTA that merges the parts, which sets the header's epoch to that search's
// when it has left the bound for the next.  kRecordCtas more make the records meanwhile.  The wait is limited (`polls`);
// true: the search is over.
// Steps of about 8 us are bound by publish, ticket, merge and this wait, the first of a large front by their items.  Front of
// the GPT-3 FFN (20 searches), a launch per search that waited for the one before 264 us, steps of one kernel 202 (now 185);
// 99 random fronts 241 and 198 us; the energy-latency front of 10 816 tilings 56.5 and 55.3.
constexpr int64_t kNoBound = INT64_MIN;         // what a search leaves that found nothing

// The low half of the header's word is the bound where it has 32 bits (a capacity).  (Unrolled: twenty searches 184.5 us, as
// a plain loop 185.6.)
__device__ __forceinline__ bool await_epoch(const SearchHeader* head, uint32_t epoch, uint32_t polls, uint32_t& low) {
#pragma unroll 4
    for (uint32_t i = 0; i < polls; ++i) {
        unsigned long long now;
        asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(now) : "l"(&head->chain_epoch) : "memory");
        low = (uint32_t)now;
        if ((int32_t)((uint32_t)(now >> 32) - epoch) >= 0) return true;
    }
    return false;
}

// The end of a chained search, by all threads of the last CTA; its record is made by another (resolve_chain).
// FRONT: the least (energy, latency, block) of all CTAs is the next point of the energy-latency front.  It is left as a
// latency optimum under that energy; the next search allows one word less of latency.
// Else: the least (energy, block, buffer need); the next search allows one word of buffer less than that need.
template <bool FRONT>
__device__ __noinline__ void finalize_chain(const Plan& p, const Limits& lim, Shared& sh, ChainRecord* chain_to, uint32_t epoch,
                                            SearchHeader* __restrict__ head, const Partial* __restrict__ partials, int n_partials) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int64_t ek = kInfKey, el = kInfKey;
    uint64_t ei = UINT64_MAX;
    unsigned long long rows = 0;
    for (int c0 = tid; c0 < n_partials; c0 += 2 * kSearchThreads) {
        longlong2 v[2], w[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int c = c0 + u * kSearchThreads;
            v[u] = w[u] = make_longlong2(kInfKey, -1ll);
            if (c < n_partials) {
                v[u] = __ldcg(&partials[c].e[0]);
                w[u] = __ldcg(&partials[c].e[1]);
                rows += __ldcg(&partials[c].feasible_rows);
            }
        }
#pragma unroll
        for (int u = 0; u < 2; ++u)
            if (triple_less(v[u].x, v[u].y, (uint64_t)w[u].x, ek, el, ei)) { ek = v[u].x; el = v[u].y; ei = (uint64_t)w[u].x; }
    }
    for (int off = 16; off; off >>= 1) rows += __shfl_down_sync(kFull, rows, off);
    warp_min_triple(ek, el, ei);
    if (lane == 0) {
        sh.feasible_rows[warp] = rows;
        sh.tops[warp][0] = make_longlong2((long long)ek, (long long)el);
        sh.tops[warp][1] = make_longlong2((long long)ei, 0);
    }
    __syncthreads();
    if (warp) return;
    rows = lane < kWarps ? sh.feasible_rows[lane] : 0;
    for (int off = kWarps / 2; off; off >>= 1) rows += __shfl_down_sync(kFull, rows, off);
    ek = sh.tops[lane & (kWarps - 1)][0].x;
    el = sh.tops[lane & (kWarps - 1)][0].y;
    ei = (uint64_t)sh.tops[lane & (kWarps - 1)][1].x;
    warp_min_triple(ek, el, ei);
    const bool found = ek != kInfKey;
    if (lane == 0) {
        const unsigned long long fit = rows * p.n_sm;
        if (FRONT) *chain_to = {(long long)(found ? el : kInfKey), (unsigned long long)ei, fit, (long long)ek, 0, 0};
        else *chain_to = {(long long)ek, (unsigned long long)el, fit, (long long)lim.cap_words, (long long)ei, 0};
        const int64_t bound = !found ? kNoBound : (FRONT ? el : (int64_t)ei) - 1;
        const unsigned long long word = (unsigned long long)epoch << 32 | (found ? (uint32_t)bound : 0xffffffffu);
        head->chain_bound = bound;
        head->done_ctas = 0;
        asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(&head->chain_epoch), "l"(word) : "memory");
    }
}

// Run by every thread of ONE CTA (the last one to finish) after all CTAs have published their partial lists.
template <int OBJ, int MODE>
__device__ __noinline__ void finalize_step(const Plan& p, const Limits& lim, Shared& sh, SearchHeader* __restrict__ head,
                                           const Partial* __restrict__ partials, int n_partials,
                                           mmee_result_t* __restrict__ out_best, mmee_result_t* __restrict__ out_topk) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr bool MULTI = MODE == kModeMulti;
    const int k = MULTI ? (int)p.topk : 1;
    int64_t ek = kInfKey;
    uint64_t ei = UINT64_MAX;
    unsigned long long rows = 0, live = 0;

    // ---- the k best items of all CTAs (loads bypass the L1 cache, both of a thread's in flight at once: BERT 8.78 us with
    // one after the other, 8.72 so, pruned sweep 10.15 and 10.03, register-file BERT 20.29 and 20.03)
    for (int c0 = 0; c0 < n_partials; c0 += 2 * kSearchThreads) {
        longlong2 firsts[2], tails[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int c = c0 + u * kSearchThreads + tid;
            firsts[u] = make_longlong2(kInfKey, -1ll);
            tails[u] = make_longlong2(0, 0);
            if (c < n_partials) {
                firsts[u] = __ldcg(&partials[c].e[0]);
                tails[u] = __ldcg(reinterpret_cast<const longlong2*>(&partials[c].count));
            }
        }
#pragma unroll 1
        for (int u = 0; u < 2; ++u) {
            const longlong2 first = u ? firsts[1] : firsts[0], tail = u ? tails[1] : tails[0];
            const uint32_t count = (uint32_t)tail.x;
            live += (uint64_t)tail.x >> 32;
            rows += (unsigned long long)tail.y;
            if (!MULTI) {
                if (count && pair_less(first.x, (uint64_t)first.y, ek, ei)) { ek = first.x; ei = (uint64_t)first.y; }
                continue;
            }
            // the lists of this warp's lanes, best heads first: once a head does not precede the k-th entry, no
            // other list adds anything
            int64_t hk = count ? first.x : kInfKey;
            uint64_t hi = count ? (uint64_t)first.y : UINT64_MAX;
            while (true) {
                int64_t bk = hk;
                uint64_t bi = hi;
                warp_min_pair(bk, bi);
                if (!pair_less(bk, bi, __shfl_sync(kFull, ek, k - 1), __shfl_sync(kFull, ei, k - 1))) break;
                const int src = __ffs(__ballot_sync(kFull, hk == bk && hi == bi && count)) - 1;
                const int n = (int)__shfl_sync(kFull, count, src);
                longlong2 theirs = make_longlong2(kInfKey, -1ll);
                if (lane < n) theirs = __ldcg(&partials[c0 + u * kSearchThreads + warp * 32 + src].e[lane]);
                reg_merge(ek, ei, k, theirs.x, (uint64_t)theirs.y, lane);
                if (lane == src) { hk = kInfKey; hi = UINT64_MAX; }
            }
        }
    }
    for (int off = 16; off; off >>= 1) {
        rows += __shfl_down_sync(kFull, rows, off);
        live += __shfl_down_sync(kFull, live, off);
    }
    if (lane == 0) {
        sh.feasible_rows[warp] = rows;
        sh.live_tilings[warp] = (uint32_t)live;
    }
    int found;
    uint32_t n_groups = 0;         // groups of five rows of the blocks evaluated mapping by mapping
    int64_t bound;
    if (!MULTI) {
        warp_min_pair(ek, ei);
        min_over_warps(sh, lane, warp, ek, ei);
        found = ek != kInfKey ? 1 : 0;
        bound = ek;
        // ---- the winning block, mapping by mapping
        const int item = split_item(warp, lane);
        if (found && item >= 0) block_item(p, SharedDivisors{sh}, (uint32_t)ei, item, &sh.block[0]);
        __syncthreads();
        if (found) {
            n_groups = block_rows(sh.block[0]) / 5u;
            best_of_block<OBJ, false>(p, lim, sh, bound, 0, ek, ei);
        }
        min_over_warps(sh, lane, warp, ek, ei);
    } else {
        merge_warps(sh, k, lane, warp, ek, ei);
        const longlong2 e = lane < kTopK ? sh.tops[0][lane] : make_longlong2(kInfKey, -1ll);
        found = __popc(__ballot_sync(kFull, e.x != kInfKey));
        bound = found == k ? (int64_t)__shfl_sync(kFull, e.x, k - 1) : kInfKey - 1;     // k items hold k mappings
        const unsigned same = __match_any_sync(kFull, (unsigned long long)e.y);      // (by all lanes, whatever they hold)
        const bool fresh = e.x != kInfKey && __ffs(same) - 1 == lane;                 // the first item of its block
        unsigned m = __ballot_sync(kFull, fresh);
        const int n_fresh = __popc(m);
        ek = kInfKey;
        ei = UINT64_MAX;
        int64_t lk = kInfKey;           // the k-th best mapping so far
        uint64_t li = UINT64_MAX;
        __syncthreads();                // sh.tops has been read
        // ---- the winning blocks, mapping by mapping, best block first; once a block's (least key, first index) does
        // not precede the k-th mapping, neither does a later one's.  (Usually the first block is the only one: its
        // tables are built by three warps, the others' one block to a warp.)
        bool more = true;
        for (int j0 = 0; more && j0 < n_fresh; j0 += j0 ? kWarps : 1) {
            const int n_batch = j0 ? min(kWarps, n_fresh - j0) : 1;
            const int next = __ffs(m) - 1;
            const int64_t next_key = __shfl_sync(kFull, e.x, next);
            const uint32_t next_id = (uint32_t)__shfl_sync(kFull, e.y, next);
            if (!pair_less(next_key, block_first_idx(p, next_id), lk, li)) break;
            int64_t bk[kWarps];
#pragma unroll
            for (int j = 0; j < kWarps; ++j) {
                if (j >= n_batch) continue;
                const int src = __ffs(m) - 1;
                m &= m - 1;
                bk[j] = __shfl_sync(kFull, e.x, src);
                const uint32_t id = (uint32_t)__shfl_sync(kFull, e.y, src);
                const int item = j0 ? (j == warp ? lane : -1) : split_item(warp, lane);
                if (item >= 0) block_item(p, SharedDivisors{sh}, id, item, &sh.block[j]);
            }
            if (lane == 0) sh.kth[warp] = kInfKey;
            __syncthreads();
#pragma unroll 1
            for (int j = 0; j < n_batch; ++j) {
                int64_t key = bk[0];
#pragma unroll
                for (int i = 1; i < kWarps; ++i) key = i == j ? bk[i] : key;
                more = pair_less(key, sh.block[j].first_idx, lk, li);
                if (!more) break;
                n_groups += block_rows(sh.block[j]) / 5u;
                best_of_block_multi<OBJ>(p, lim, sh, j, bound, k, lane, lk, li, ek, ei);
                merge_warps(sh, k, lane, warp, ek, ei);
                const longlong2 last = sh.tops[0][k - 1];
                lk = last.x;
                li = (uint64_t)last.y;
                if (warp) { ek = kInfKey; ei = UINT64_MAX; }        // (warp 0 goes on with the merged list)
                __syncthreads();
            }
        }
        if (!n_fresh && lane < kTopK && warp == 0) sh.tops[0][lane] = make_longlong2(kInfKey, -1ll);
        __syncthreads();
    }

    // ---- every winner evaluated in full by its lanes (a warp, or half a warp per record when there are several); the
    // key it was ranked by must be the key of that evaluation, or the records are marked as no result
    constexpr int kLanes = MULTI ? 16 : 32;
    constexpr int kWords = sizeof(mmee_result_t) / 8;
    static_assert(sizeof(mmee_result_t) % 8 == 0 && MMEE_MAX_TOPK == 2 * kWarps, "two records to a warp");
    const int rec = MULTI ? 2 * warp + (lane >> 4) : 0, l = lane & (kLanes - 1);
    longlong2 entry = make_longlong2(kInfKey, -1ll);
    if (MULTI && lane < k) entry = sh.tops[0][lane];
    const int n_out = MULTI ? __popc(__ballot_sync(kFull, entry.x != kInfKey)) : (ek != kInfKey ? 1 : 0);
    if (tid == 0 && (n_out == 0) != (found == 0)) atomicOr(&sh.check_failed, 1u);
    if (MULTI ? 2 * warp < k : warp == 0) {
        mmee_result_t& r = sh.record[rec];          // put together in shared memory and copied from there
        const int64_t rk = MULTI ? (int64_t)__shfl_sync(kFull, entry.x, rec) : ek;
        uint64_t ri = MULTI ? (uint64_t)__shfl_sync(kFull, entry.y, rec) : ei;
        const uint64_t other = MULTI ? (uint64_t)__shfl_sync(kFull, entry.y, 2 * warp) : ei;
        const bool full = rec < n_out;
        if (!full) ri = other;                      // (a half without a record goes along with the other)
        if ((MULTI ? 2 * warp : 0) < n_out)
            evaluate_candidate_lanes<kLanes>(p, SharedDivisors{sh}, ri, lim.cap_words, lane, full, r);
        if (full) {
            if (l == 0) {
                const int64_t key = OBJ == MMEE_OBJ_EDP ? __double_as_longlong(r.edp_key) : key_of<OBJ>(r.e_key, r.l_key, lim.key_cap);
                if (!(key == rk && r.feasible && r.t >= p.t_begin && r.t < p.t_end)) atomicOr(&sh.check_failed, 1u);
            }
        } else {
            // empty slot
            unsigned long long* raw = reinterpret_cast<unsigned long long*>(&r);
            for (int i = l; i < kWords; i += kLanes) raw[i] = 0;
            __syncwarp(MULTI ? 0xffffu << (lane & 16) : kFull);
            if (l == 0) {
                r.idx = MMEE_NO_INDEX;
                r.status = n_out ? MMEE_OK : MMEE_ERR_NO_FEASIBLE;
            }
        }
        __syncwarp();
        if (out_topk && rec < k) {
            const unsigned long long* from = reinterpret_cast<const unsigned long long*>(&r);
            unsigned long long* to = reinterpret_cast<unsigned long long*>(&out_topk[rec]);
            for (int i = l; i < kWords; i += kLanes) to[i] = from[i];
        }
    }
    __syncthreads();
    if (warp == 0) {
        unsigned long long all_rows = lane < kWarps ? sh.feasible_rows[lane] : 0;
#pragma unroll
        for (int off = kWarps / 2; off; off >>= 1) all_rows += __shfl_xor_sync(kFull, all_rows, off);
        mmee_result_t& best = sh.record[0];
        if (lane == 0) {
            best.n_total = (p.t_end - p.t_begin) * (uint64_t)p.rows_per_tiling * 9u;
            best.n_feasible = all_rows * (uint64_t)p.n_sm;
            if (sh.check_failed) best.status = MMEE_ERR_CHECK;
        }
        __syncwarp();
        const unsigned long long* from = reinterpret_cast<const unsigned long long*>(&best);
        unsigned long long* to = reinterpret_cast<unsigned long long*>(out_best);
        for (int i = lane; i < kWords; i += 32) to[i] = from[i];
    } else if (tid == 32) {
        // ready for the next search on this scratch
        unsigned long long all_live = 0;
        for (int w = 0; w < kWarps; ++w) all_live += sh.live_tilings[w];
        head->G = kInfKey - 1;
        head->last_exact_groups = n_groups;
        const uint32_t unfused_modes = (p.fuse_mask >> 1 & 1u) + (p.fuse_mask >> 2 & 1u);
        head->last_tested_rows = all_live * p.n_orders * ((p.fuse_mask & 1u ? kFusedReps : 0u) + (unfused_modes ? 18u : 0u));
        head->done_ctas = 0;
    }
}

// The full record of an optimum, by one CTA after load_shared: the first mapping with key `key` of block `where`.  key
// kInfKey: nothing fits.
// STAIRS: the first one that also has the buffer need `need`, the least of them.  A search that returns the first mapping
// with the least key and then searches on with one word less than that mapping's need would meet those with larger needs
// before it: the record's n_feasible is the number of mappings that fit under the last bound of such a sequence.  Where
// that is not the bound this one was found under, reserved2[0] says what it is, plus one (a rare case: index order
// raises needs), and the caller searches there.
template <int OBJ, bool STAIRS>
__device__ __forceinline__ void resolve_record(const Plan& p, const Limits& lim, Shared& sh,
                                               int64_t key, uint64_t where, unsigned long long n_feasible, int64_t need,
                                               mmee_result_t* out) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    mmee_result_t& r = sh.record[0];
    uint32_t before_need = 0;
    if (key != kInfKey) {
        int64_t ek = kInfKey;
        uint64_t ei = UINT64_MAX;
        uint64_t before = UINT64_MAX;           // STAIRS: least need of a mapping with that key before the one found
        const int item = split_item(warp, lane);
        if (item >= 0) block_item(p, SharedDivisors{sh}, (uint32_t)where, item, &sh.block[0]);
        __syncthreads();
        if (STAIRS) {
            best_of_block<OBJ, true>(p, lim, sh, key, need, ek, ei);
            min_over_warps(sh, lane, warp, ek, ei);
            before = least_need_before<OBJ>(p, lim, sh, key, ei);
            int64_t zero = 0;
            min_over_warps(sh, lane, warp, zero, before);
        } else {
            best_of_block<OBJ, false>(p, lim, sh, key, 0, ek, ei);
            min_over_warps(sh, lane, warp, ek, ei);
        }
        if (before != UINT64_MAX) before_need = (uint32_t)before;
        if (warp == 0) {
            const bool have = ek == key;
            evaluate_candidate_lanes<32>(p, SharedDivisors{sh}, have ? ei : 0, lim.cap_words, lane, lane == 0, r);
            if (lane == 0) {
                const int64_t own = OBJ == MMEE_OBJ_EDP ? __double_as_longlong(r.edp_key) : key_of<OBJ>(r.e_key, r.l_key, lim.key_cap);
                if (!(have && own == key && r.feasible && r.t >= p.t_begin && r.t < p.t_end)) r.status = MMEE_ERR_CHECK;
            }
        }
    } else if (warp == 0) {
        unsigned long long* raw = reinterpret_cast<unsigned long long*>(&r);
        for (int i = lane; i < (int)(sizeof(r) / 8); i += 32) raw[i] = 0;
        __syncwarp();
        if (lane == 0) {
            r.idx = MMEE_NO_INDEX;
            r.status = MMEE_ERR_NO_FEASIBLE;
        }
    }
    if (warp == 0) {
        if (lane == 0) {
            r.n_total = (p.t_end - p.t_begin) * (uint64_t)p.rows_per_tiling * 9u;
            r.n_feasible = n_feasible;
            if (STAIRS) r.reserved2[0] = before_need;
        }
        __syncwarp();
        const unsigned long long* from = reinterpret_cast<const unsigned long long*>(&r);
        unsigned long long* to = reinterpret_cast<unsigned long long*>(out);
        for (int i = lane; i < (int)(sizeof(r) / 8); i += 32) to[i] = from[i];
    }
}

// The records of chained searches as they end, by kRecordCtas CTAs, this one number `which`: the first search has the epoch
// shape.chain_epoch, the last one finds nothing.  A record is written as a whole or not at all.
template <bool FRONT>
__device__ __noinline__ void resolve_chain(const Plan& p, const LaunchShape& shape, Shared& sh, const SearchHeader* head, uint32_t which,
                                           mmee_result_t* out) {
    for (uint32_t i = 0; i < shape.chain_steps; ++i) {
        __syncthreads();
        uint32_t low;
        if (threadIdx.x == 0) sh.waited = await_epoch(head, shape.chain_epoch + i, shape.chain_polls, low) ? 1u : 0u;
        __syncthreads();
        if (!sh.waited) return;
        const volatile ChainRecord* from = shape.chain_to + i;
        const ChainRecord c = {from->key, from->where, from->n_feasible, from->bound, from->need, 0};
        if (i % kRecordCtas == which) {
            if (FRONT) resolve_record<MMEE_OBJ_LATENCY_ECAP, false>(p, Limits{p.cap_words, c.bound}, sh, c.key, c.where, c.n_feasible, 0, out + i);
            else resolve_record<MMEE_OBJ_ENERGY, true>(p, Limits{c.bound, 0}, sh, c.key, c.where, c.n_feasible, c.need, out + i);
        }
        if (c.key == kInfKey) return;
    }
}

// ------------------------------------------------------------------------------------------------
// the search kernel
// ------------------------------------------------------------------------------------------------

// Searches launched one after the other overlap (programmatic dependent launch), in one of two ways.
//   early: a search lets the next one start at once; that one's CTAs move in as this one's leave, and wait for its end
//          before they publish, since it may still use their scratch;
//   late:  only the CTA that finalizes waits for the kernel before, and lets the next search start after that wait.  The
//          CTAs then publish while the search before finalizes, into the other one of the handle's two scratches: the
//          search that used theirs last had ended before the one before them let them start.  (Always for k > 1, whose CTAs
//          share a bound through the scratch while they work on their items.)
// A kernel that is not launched this way follows a search as usual, and a search follows one as usual.  Searches one after
// the other, without and with this (us each): smallest configuration 20.5 and 8.9, BERT energy 22.9 and 10.4, GQA latency
// 28.7 and 13.7, convolution chain top-16 133 and 58 (other changes between them included).
__device__ __forceinline__ void release_next_kernel() { asm volatile("griddepcontrol.launch_dependents;"); }
__device__ __forceinline__ void wait_previous_kernel() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// The number of CTAs that drew a ticket before; what they wrote before that is visible from here on, and what the calling
// warp has written is to those that draw one later.
__device__ __forceinline__ uint32_t draw_ticket(unsigned int* count) {
    uint32_t n;
    asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(n) : "l"(count) : "memory");
    return n;
}

// The tables of one tiling, by eight threads (sub = 0..7) once tb->b is there: one stationary mode of one operator each,
// and the sizes between them.
template <bool TERMS>
__device__ __forceinline__ void build_tile(const Plan& p, const Shared& sh, const uint32_t b[8], uint32_t t, int sub, TileTab* tb) {
    if (TERMS && sub < 6) {
        const int op = sub >= 3 ? 1 : 0, sm = sub - 3 * op;
        int64_t P, Q;
        stationary_terms(p, SharedDivisors{sh}, b, op, sm, P, Q);
        (op ? tb->st.P2 : tb->st.P1)[sm] = P;
        (op ? tb->st.Q2 : tb->st.Q1)[sm] = Q;
    }
    for (int i = sub; i < kSizeSlots; i += 8) tb->size[i] = sat_size(size_words(p.dim, tb->b + 4, i));
    if (sub == 7) tb->t = t;
}

template <int OBJ, int MODE>
__global__ void __launch_bounds__(kSearchThreads, 2)
search_kernel(const __grid_constant__ Plan p, const LaunchShape shape, SearchHeader* __restrict__ head, Partial* __restrict__ partials,
              mmee_result_t* __restrict__ out_best, mmee_result_t* __restrict__ out_topk) {
    constexpr bool PRUNE = MODE == kModePrune, MULTI = MODE == kModeMulti, CHAIN = MODE == kModeChain;
    constexpr bool ARRAYS = MODE == kModeArrays;
    constexpr bool FRONT = CHAIN && OBJ == MMEE_OBJ_ENERGY_LCAP;      // least (energy, latency) under a bound on the latency
    constexpr bool STAIRS = CHAIN && OBJ == MMEE_OBJ_ENERGY;          // least (energy, block, buffer need) under a capacity
    static_assert(FRONT || STAIRS || !CHAIN, "only the searches of the Pareto fronts are chained");
    __shared__ Shared sh;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool late = MULTI || shape.late;
    if (!late) release_next_kernel();
    load_shared<PRUNE>(p, p.pe_rows, p.pe_cols, sh);
    // Array shapes: the stationary-pair terms of shape y and tiling slot i at [y * chunk + i], behind the tilings' tables;
    // the warps' best items of shape y in sh.tops[.][y].
    StatTerms* terms = reinterpret_cast<StatTerms*>(&sh.tile[shape.chunk]);
    if (ARRAYS && tid < kWarps * (int)MMEE_MAX_TOPK) sh.tops[tid / (int)MMEE_MAX_TOPK][tid % (int)MMEE_MAX_TOPK] = make_longlong2(kInfKey, -1ll);
    // STAIRS: the table slots of the tilings that fit under the bound, where the kept rows of the other modes lie.
    uint8_t* fit_slots = reinterpret_cast<uint8_t*>(&sh.kept);
    static_assert(kMaxChunk <= 256 && kMaxChunk <= sizeof(KeptMasks), "one byte per table");
    if (tid == 0) {
        sh.n_live = sh.n_fit = 0;
        sh.cursor = 0;
        sh.check_failed = 0;
    }
    __syncthreads();

    if (CHAIN && blockIdx.x >= shape.grid) {
        resolve_chain<FRONT>(p, shape, sh, head, blockIdx.x - shape.grid, out_topk);
        return;
    }

    const int k = MULTI ? (int)p.topk : 1;
    const int64_t I = p.dim[0], K = p.dim[1], L = p.dim[2], J = p.dim[3];
    const DimWords dw = {I * K, K * L, L * J, I * J, I * L};
    Limits lim = {p.cap_words, p.key_cap};
    int capc = (int)p.cap_words;
    const uint32_t grid = CHAIN ? shape.grid : gridDim.x, n_tilings = (uint32_t)(p.t_end - p.t_begin);
    const uint32_t n_orders = p.n_orders;
    auto any = [](bool v) { return __any_sync(kFull, v) != 0; };

    // the best item so far: k = 1 of this thread, else the warp's list (lane j holds entry j)
    int64_t ek = kInfKey;
    uint64_t ei = UINT64_MAX;
    int64_t el = kInfKey;           // FRONT: its latency.  STAIRS: (el, ei) are the block and its need
    unsigned long long my_rows = 0;
    uint32_t my_live = 0;

    auto offer = [&](int64_t key, uint32_t id, bool valid) {
        if (!MULTI) {
            if (valid && pair_less(key, id, ek, ei)) { ek = key; ei = id; }
            return;
        }
        const int64_t lk = __shfl_sync(kFull, ek, k - 1);
        const uint64_t li = __shfl_sync(kFull, ei, k - 1);
        const bool pend = valid && key != kInfKey && key <= *reinterpret_cast<volatile long long*>(&sh.G) && pair_less(key, id, lk, li);
        if (!__any_sync(kFull, pend)) return;
        warp_offer(ek, ei, k, key, id, pend, lane);
        // a full list bounds the k-th smallest key for everybody
        if (lane == k - 1 && ek < *reinterpret_cast<volatile long long*>(&sh.G)) {
            atomicMin(&sh.G, (long long)ek);
            atomicMin(&head->G, (long long)ek);
        }
    };

    // FRONT: the item's least (energy, latency) over the stationary pairs; pair(s, e, l) forms those of pair s.
    auto offer_front = [&](auto pair, uint32_t id, bool valid) {
        int64_t be = kInfKey, bl = kInfKey;
#pragma unroll
        for (int s = 0; s < 9; ++s) {
            int64_t e, l;
            pair(s, e, l);
            const bool better = ((p.sm_mask >> s) & 1u) && l <= lim.key_cap && (e < be || (e == be && l < bl));
            be = better ? e : be;
            bl = better ? l : bl;
        }
        if (valid && triple_less(be, bl, id, ek, el, ei)) { ek = be; el = bl; ei = id; }
    };

    auto offer_stairs = [&](int64_t key, uint32_t id, int need, bool valid) {
        if (valid && triple_less(key, (int64_t)id, (uint64_t)need, ek, el, ei)) { ek = key; el = id; ei = (uint64_t)need; }
    };

    // The same for every array shape, one after the other: key_of_terms(terms) is the item's least key.
    auto offer_arrays = [&](auto key_of_terms, uint32_t slot, uint32_t id, bool valid) {
        for (uint32_t y = 0; y < shape.n_arrays; ++y) {
            const int64_t key = key_of_terms(terms[y * shape.chunk + slot]);
            const longlong2 own = sh.tops[warp][y];
            const bool better = valid && pair_less(key, id, own.x, (uint64_t)own.y);
            if (!any(better)) continue;
            int64_t nk = better ? key : kInfKey;
            uint64_t ni = better ? id : UINT64_MAX;
            warp_min_pair(nk, ni);
            if (lane == 0) sh.tops[warp][y] = make_longlong2((long long)nk, (long long)ni);
            __syncwarp();
        }
    };

    const bool one_pass = (uint64_t)shape.chunk * grid >= n_tilings;        // chained: the tables stay
    for (uint32_t step = 0;; ++step) {
        if (CHAIN && (step || shape.chain_read)) {
            __syncthreads();                // the counters of the search before are no longer in use
            if (tid == 0) {
                uint32_t low = 0;
                const bool over = !step || await_epoch(head, shape.chain_epoch + step - 1, shape.chain_polls, low);
                if (!over) sh.bound = kNoBound;
                else if (step && STAIRS) sh.bound = low == 0xffffffffu ? kNoBound : (int64_t)low;
                else sh.bound = *reinterpret_cast<volatile long long*>(&head->chain_bound);
                sh.n_fit = sh.cursor = 0;
                if (!one_pass) sh.n_live = 0;
            }
            __syncthreads();
            const int64_t bound = sh.bound;
            if (bound == kNoBound) return;
            if (OBJ == MMEE_OBJ_ENERGY) {
                lim.cap_words = bound;
                capc = (int)bound;
            } else {
                lim.key_cap = bound;
            }
            ek = el = kInfKey;
            ei = UINT64_MAX;
            my_rows = 0;
        }
        // Tiling number m of this CTA is one of the m-th `grid` consecutive ones, a different one in every round (a fixed
        // one would be the same divisor of the last dimension again and again).
        for (uint32_t m0 = 0; (uint64_t)m0 * grid < n_tilings; m0 += shape.chunk) {
            if (m0) {
                __syncthreads();                // the previous pass's tables are no longer in use
                if (tid == 0) { sh.n_live = sh.n_fit = 0; sh.cursor = 0; }
                __syncthreads();
            }
            for (uint32_t j0 = 0; j0 < (step && one_pass ? 0 : shape.chunk); j0 += kSearchThreads / 8) {
                const uint32_t j = j0 + (uint32_t)tid / 8u, m = m0 + j;
                uint64_t rel = (uint64_t)m * grid;
                const bool mine = j < shape.chunk && rel < n_tilings;
                rel += (blockIdx.x + m) % grid;
                uint32_t b[8], t = 0;
                bool live = mine && rel < n_tilings;
                if (live) {
                    t = (uint32_t)(p.t_begin + rel);
                    tiling_bounds(p, SharedDivisors{sh}, t, b);
                    // With every operand at L3 the buffer need is smallest: max(A+B+C, C+D+E) tiles (Eq. 1-4).
                    const uint64_t ta = (uint64_t)b[4] * b[5], tbb = (uint64_t)b[5] * b[6], tc = (uint64_t)b[4] * b[6];
                    const uint64_t td = (uint64_t)b[6] * b[7], te = (uint64_t)b[4] * b[7];
                    live = ta + tbb + tc <= (uint64_t)capc && tc + td + te <= (uint64_t)capc;
                }
                uint32_t slot = 0;
                if (live && (tid & 7) == 0) slot = atomicAdd(&sh.n_live, 1u);
                slot = __shfl_sync(kFull, slot, lane & ~7);
                if (live) {
                    uint32_t own = b[0];
    #pragma unroll
                    for (int d = 1; d < 8; ++d) own = (tid & 7) == d ? b[d] : own;
                    sh.tile[slot].b[tid & 7] = own;
                }
                __syncwarp();
                if (live) build_tile<!ARRAYS>(p, sh, b, t, tid & 7, &sh.tile[slot]);
            }
            if (MULTI && m0 == 0 && tid == 0) sh.G = *reinterpret_cast<volatile long long*>(&head->G);
            __syncthreads();
            if (ARRAYS) {
                const uint32_t n_live = sh.n_live;
                for (uint32_t i = tid; i < n_live * 6u * shape.n_arrays; i += kSearchThreads) {
                    const uint32_t y = i / (n_live * 6u), u = i - y * n_live * 6u, slot = u / 6u;
                    const int op = u - slot * 6u >= 3u ? 1 : 0, sm = (int)(u - slot * 6u) - 3 * op;
                    StatTerms& st = terms[y * shape.chunk + slot];
                    int64_t P, Q;
                    stationary_terms(p, ArrayDivisors{sh, shape.array[y][0], shape.array[y][1]}, sh.tile[slot].b, op, sm, P, Q);
                    (op ? st.P2 : st.P1)[sm] = P;
                    (op ? st.Q2 : st.Q1)[sm] = Q;
                }
                __syncthreads();
            }

            if (STAIRS) {
                // The tables are those of the bound the plan has.  (Front of the GPT-3 FFN, twenty searches: 281 us with
                // items for every table, 263 with this.)
                if ((uint32_t)tid < sh.n_live) {
                    const uint32_t* b = sh.tile[tid].b;
                    const uint64_t tc = (uint64_t)b[4] * b[6];
                    const uint64_t first = (uint64_t)b[4] * b[5] + (uint64_t)b[5] * b[6], second = (uint64_t)b[6] * b[7] + (uint64_t)b[4] * b[7];
                    if (tc + max(first, second) <= (uint64_t)capc) fit_slots[atomicAdd(&sh.n_fit, 1u)] = (uint8_t)tid;
                }
                __syncthreads();
            }
            const uint32_t n_tiles = STAIRS ? sh.n_fit : sh.n_live, per_class = n_tiles * n_orders;
            if (tid == 0) my_live += n_tiles;
            const uint32_t fused_items = (p.fuse_mask & 1u) ? 3u * per_class : 0u;
            const uint32_t fused_groups = (fused_items + 31u) / 32u;
            const uint32_t groups = fused_groups + ((p.fuse_mask & 6u) ? (per_class + 31u) / 32u : 0u);
            while (true) {
                uint32_t g = 0;
                if (lane == 0) g = atomicAdd(&sh.cursor, 1u);
                g = __shfl_sync(kFull, g, 0);
                if (g >= groups) break;
                long long g_seen = 0;       // k > 1: the other CTAs' bound, used after this item
                if (MULTI && lane == 0) g_seen = *reinterpret_cast<volatile long long*>(&head->G);
                const bool fused = g < fused_groups;
                uint32_t i = (fused ? g : g - fused_groups) * 32u + (uint32_t)lane;
                const uint32_t n_items = fused ? fused_items : per_class;
                const bool valid = i < n_items;
                i = valid ? i : n_items - 1;
                uint32_t c = 0;
                if (fused) {
                    c = i >= 2u * per_class ? 2u : (i >= per_class ? 1u : 0u);
                    i -= c * per_class;
                }
                uint32_t slot = n_orders == 6u ? i / 6u : i / 2u;
                const uint32_t os = i - slot * n_orders;
                if (STAIRS) slot = fit_slots[slot];
                const TileTab& tb = sh.tile[slot];
                const OrderInfo& oi = sh.order[os];
                const uint32_t id = tb.t * p.n_blocks + os;
                if (fused) {
                    uint32_t rows;
                    int64_t x;
                    int need;
                    fused_class<PRUNE, STAIRS>(tb, oi, dw, (int)c, capc, PRUNE ? sh.kept.fused[os][c] : nullptr, any, rows, x, need);
                    if (valid) my_rows += rows;
                    const bool some = valid && x < kNoRow;
                    if (any(some)) {
                        const int64_t y = some ? x : 0, rho = oi.recompute[c] != 0 ? (int64_t)tb.b[LOOP_J] : 1;
                        auto key = [&](const StatTerms& t) { return fused_least_key<OBJ>(t, y, rho, p.sm_mask, p.c_dram_gb, lim.key_cap); };
                        auto pair = [&](int s, int64_t& e, int64_t& l) {
                            e = p.c_dram_gb * y + tb.st.P1[s / 3] * rho + tb.st.P2[s % 3];
                            l = max64(y, tb.st.Q1[s / 3] * rho + tb.st.Q2[s % 3]);
                        };
                        if (ARRAYS) offer_arrays(key, slot, id, some);
                        else if (FRONT) {
                            // No mapping of the item is faster than this; after the first search few are fast enough
                            // (front of 10 816 tilings, one point: 53.9 us without this test, 52.5 with it).
                            const bool can = some && max64(y, min3(tb.st.Q1) * rho + min3(tb.st.Q2)) <= lim.key_cap;
                            if (any(can)) offer_front(pair, id, can);
                        }
                        else if (STAIRS) offer_stairs(key(tb.st), id, need, some);
                        else offer(key(tb.st), id, some);
                    }
                } else {
                    uint32_t fit1, fit2, rows;
                    int64_t x1, x2;
                    int need;
                    unfused_nests<PRUNE, STAIRS>(tb, oi, dw, capc, fit1, fit2, rows, x1, x2, need);
                    const bool some = valid && x1 < kNoRow;
                    if (!any(some)) continue;
                    const int64_t y1 = some ? x1 : 0, y2 = some ? x2 : 0;
                    uint32_t block = p.n_fused_blocks;
    #pragma unroll
                    for (int phi = 1; phi <= 2; ++phi) {
                        if (!((p.fuse_mask >> phi) & 1u)) continue;
                        if (PRUNE) {
                            rows = 0;
                            for (int ab = 0; ab < 9; ++ab)
                                if ((fit1 >> ab) & 1u) rows += (uint32_t)__popc(fit2 & sh.kept.unfused[phi - 1][os][ab]);
                        }
                        if (some) my_rows += rows;
                        const int64_t pass = phi == 2 ? 2 * dw.il : 0;
                        auto key = [&](const StatTerms& t) { return unfused_least_key<OBJ>(t, y1, y2, pass, p.sm_mask, p.c_dram_gb, lim.key_cap); };
                        auto pair = [&](int s, int64_t& e, int64_t& l) {
                            e = p.c_dram_gb * (y1 + y2 + pass) + tb.st.P1[s / 3] + tb.st.P2[s % 3];
                            l = max64(y1, tb.st.Q1[s / 3]) + pass + max64(y2, tb.st.Q2[s % 3]);
                        };
                        if (ARRAYS) offer_arrays(key, slot, id + block, some);
                        else if (FRONT) {
                            const bool can = some && max64(y1, min3(tb.st.Q1)) + pass + max64(y2, min3(tb.st.Q2)) <= lim.key_cap;
                            if (any(can)) offer_front(pair, id + block, can);
                        }
                        else if (STAIRS) offer_stairs(key(tb.st), id + block, need, some);
                        else offer(key(tb.st), id + block, some);
                        block += n_orders;
                    }
                }
                if (MULTI && lane == 0 && g_seen < sh.G) atomicMin(&sh.G, g_seen);
            }
        }

        // ---- this CTA's result
        for (int off = 16; off; off >>= 1) my_rows += __shfl_down_sync(kFull, my_rows, off);
        if (lane == 0) sh.feasible_rows[warp] = my_rows;
        if (MULTI) {
            merge_warps(sh, k, lane, warp, ek, ei);
        } else if (CHAIN) {
            warp_min_triple(ek, el, ei);
            if (lane == 0) {
                sh.tops[warp][0] = make_longlong2((long long)ek, (long long)el);
                sh.tops[warp][1] = make_longlong2((long long)ei, 0);
            }
            __syncthreads();
        } else if (!ARRAYS) {
            warp_min_pair(ek, ei);
            if (lane == 0) sh.tops[warp][0] = make_longlong2((long long)ek, (long long)ei);
            __syncthreads();
        }
        if (!late && !CHAIN) wait_previous_kernel();        // from here on the scratch is touched
        if (ARRAYS) {
            // the best item of every shape; the kernel that follows merges them (resolve_arrays_kernel)
            __syncthreads();
            Partial* out = &partials[blockIdx.x];
            for (uint32_t y = warp; y < shape.n_arrays; y += kWarps) {
                const longlong2 v = sh.tops[lane & (kWarps - 1)][y];
                int64_t nk = v.x;
                uint64_t ni = (uint64_t)v.y;
                warp_min_pair(nk, ni);
                if (lane == 0) out->e[y] = make_longlong2((long long)nk, (long long)ni);
            }
            if (tid == 0) {
                unsigned long long rows = 0;
                for (int w = 0; w < kWarps; ++w) rows += sh.feasible_rows[w];
                out->feasible_rows = rows;
            }
            return;
        }
        if (warp == 0) {
            Partial* out = &partials[blockIdx.x];
            uint32_t count;
            if (MULTI) {
                // an entry above the bound (some full list's last key) is not among the k best
                long long g_end = lane == 0 ? *reinterpret_cast<volatile long long*>(&head->G) : 0;
                g_end = __shfl_sync(kFull, g_end, 0);
                count = (uint32_t)__popc(__ballot_sync(kFull, ek != kInfKey && ek <= g_end));
                if (lane < (int)max(count, 1u)) out->e[lane] = make_longlong2((long long)ek, (long long)ei);
            } else if (CHAIN) {
                ek = sh.tops[lane & (kWarps - 1)][0].x;
                el = sh.tops[lane & (kWarps - 1)][0].y;
                ei = (uint64_t)sh.tops[lane & (kWarps - 1)][1].x;
                warp_min_triple(ek, el, ei);
                count = 2;
                if (lane < 2) out->e[lane] = lane ? make_longlong2((long long)ei, 0) : make_longlong2((long long)ek, (long long)el);
            } else {
                const longlong2 v = sh.tops[lane & (kWarps - 1)][0];
                ek = v.x;
                ei = (uint64_t)v.y;
                warp_min_pair(ek, ei);
                count = ek != kInfKey ? 1u : 0u;
                if (lane == 0) out->e[0] = make_longlong2((long long)ek, (long long)ei);
            }
            unsigned long long rows = lane < kWarps ? sh.feasible_rows[lane] : 0;
            for (int off = kWarps / 2; off; off >>= 1) rows += __shfl_down_sync(kFull, rows, off);
            if (lane == 0) {
                out->count = count;
                out->live_tilings = my_live;
                out->feasible_rows = rows;
            }
            // Grid reduction without a wait: every CTA makes its partial list visible, then draws a ticket; the CTA that
            // draws the last one knows that all lists are there and runs the finalize step.
            __syncwarp();
            if (lane == 0) sh.last_cta = draw_ticket(&head->done_ctas) == grid - 1 ? 1u : 0u;
        }
        __syncthreads();
        if (sh.last_cta) {
            if (late) {
                wait_previous_kernel();         // from here on the result records are touched
                release_next_kernel();
            }
            if (CHAIN) finalize_chain<FRONT>(p, lim, sh, shape.chain_to + step, shape.chain_epoch + step, head, partials, (int)grid);
            else finalize_step<OBJ, MODE>(p, lim, sh, head, partials, (int)grid, out_best, out_topk);
        }
        if (!CHAIN || step + 1 == shape.chain_steps) return;
    }
}

__global__ void reset_kernel(SearchHeader* head) {
    head->G = kInfKey - 1;
    head->done_ctas = 0;
    head->chain_epoch = 0;
}

// Merge of the CTAs' best items of array shape blockIdx.x, and the record of the optimum.
template <int OBJ>
__global__ void __launch_bounds__(kSearchThreads, 2)
resolve_arrays_kernel(const __grid_constant__ Plan p, const LaunchShape shape, const Partial* partials, mmee_result_t* out) {
    __shared__ Shared sh;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    load_shared<false>(p, shape.array[blockIdx.x][0], shape.array[blockIdx.x][1], sh);
    __syncthreads();
    wait_previous_kernel();
    int64_t ek = kInfKey;
    uint64_t ei = UINT64_MAX;
    unsigned long long rows = 0;
    for (uint32_t c = tid; c < shape.grid; c += kSearchThreads) {
        const volatile Partial* from = partials + c;        // (volatile: read after the wait)
        const int64_t key = from->e[blockIdx.x].x;
        const uint64_t num = (uint64_t)from->e[blockIdx.x].y;
        rows += from->feasible_rows;
        if (pair_less(key, num, ek, ei)) { ek = key; ei = num; }
    }
    for (int off = 16; off; off >>= 1) rows += __shfl_down_sync(kFull, rows, off);
    if (lane == 0) sh.feasible_rows[warp] = rows;
    warp_min_pair(ek, ei);
    min_over_warps(sh, lane, warp, ek, ei);
    rows = 0;
    for (int w = 0; w < kWarps; ++w) rows += sh.feasible_rows[w];
    resolve_record<OBJ, false>(p, Limits{p.cap_words, p.key_cap}, sh, ek, ei, rows * p.n_sm, 0, out + blockIdx.x);
}

// A launch that may start before the kernel before it on the stream has ended (`overlap`): the kernel waits itself.
// `together`: a cooperative one instead, whose CTAs are resident at the same time.
template <class... Args>
cudaError_t launch_overlapped(bool overlap, bool together, unsigned grid, cudaStream_t st, void (*kernel)(Args...), Args... args) {
    cudaLaunchAttribute attr = {};
    if (together) {
        attr.id = cudaLaunchAttributeCooperative;
        attr.val.cooperative = 1;
    } else {
        attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr.val.programmaticStreamSerializationAllowed = 1;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kSearchThreads);
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = overlap || together ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// (only the searches of the Pareto fronts are chained)
template <int OBJ>
constexpr int chain_mode() { return OBJ == MMEE_OBJ_ENERGY || OBJ == MMEE_OBJ_ENERGY_LCAP ? kModeChain : kModeSingle; }

template <int OBJ>
cudaError_t launch_search_t(const Plan& p, const LaunchShape& shape, SearchHeader* head, Partial* partials,
                            mmee_result_t* out_best, mmee_result_t* out_topk, cudaStream_t st) {
    auto* kernel = shape.n_arrays ? search_kernel<OBJ, kModeArrays>
                   : shape.chain_steps ? (chain_mode<OBJ>() == kModeChain ? search_kernel<OBJ, chain_mode<OBJ>()> : nullptr)
                   : p.row_pruning ? search_kernel<OBJ, kModePrune>
                   : p.topk > 1    ? search_kernel<OBJ, kModeMulti> : search_kernel<OBJ, kModeSingle>;
    if (!kernel) return cudaErrorInvalidValue;
    const uint32_t grid = shape.chain_steps ? shape.grid + kRecordCtas : shape.grid;
    return launch_overlapped(shape.overlap, shape.chain_steps != 0, grid, st, kernel, p, shape, head, partials, out_best, out_topk);
}

}  // namespace

size_t search_smem_bytes() { return sizeof(Shared); }

cudaError_t launch_search(const Plan& p, const LaunchShape& shape, SearchHeader* head, Partial* partials,
                          mmee_result_t* out_best, mmee_result_t* out_topk, cudaStream_t st) {
    switch (p.objective) {
        case MMEE_OBJ_ENERGY: return launch_search_t<MMEE_OBJ_ENERGY>(p, shape, head, partials, out_best, out_topk, st);
        case MMEE_OBJ_LATENCY: return launch_search_t<MMEE_OBJ_LATENCY>(p, shape, head, partials, out_best, out_topk, st);
        case MMEE_OBJ_EDP: return launch_search_t<MMEE_OBJ_EDP>(p, shape, head, partials, out_best, out_topk, st);
        case MMEE_OBJ_ENERGY_LCAP: return launch_search_t<MMEE_OBJ_ENERGY_LCAP>(p, shape, head, partials, out_best, out_topk, st);
        default: return launch_search_t<MMEE_OBJ_LATENCY_ECAP>(p, shape, head, partials, out_best, out_topk, st);
    }
}

uint32_t search_chunk(uint32_t n_arrays) {
    return (uint32_t)(kMaxChunk * sizeof(TileTab) / (sizeof(TileTab) + n_arrays * sizeof(StatTerms)));
}

cudaError_t launch_search_arrays(const Plan& p, const LaunchShape& shape, Partial* partials, mmee_result_t* out, cudaStream_t st) {
    const cudaError_t e = launch_search(p, shape, nullptr, partials, nullptr, nullptr, st);
    if (e != cudaSuccess) return e;
    const unsigned n = shape.n_arrays;
    const Partial* from = partials;
    switch (p.objective) {
        case MMEE_OBJ_ENERGY: return launch_overlapped(true, false, n, st, resolve_arrays_kernel<MMEE_OBJ_ENERGY>, p, shape, from, out);
        case MMEE_OBJ_LATENCY: return launch_overlapped(true, false, n, st, resolve_arrays_kernel<MMEE_OBJ_LATENCY>, p, shape, from, out);
        case MMEE_OBJ_EDP: return launch_overlapped(true, false, n, st, resolve_arrays_kernel<MMEE_OBJ_EDP>, p, shape, from, out);
        case MMEE_OBJ_ENERGY_LCAP: return launch_overlapped(true, false, n, st, resolve_arrays_kernel<MMEE_OBJ_ENERGY_LCAP>, p, shape, from, out);
        default: return launch_overlapped(true, false, n, st, resolve_arrays_kernel<MMEE_OBJ_LATENCY_ECAP>, p, shape, from, out);
    }
}

cudaError_t launch_reset(SearchHeader* head, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = cfg.blockDim = dim3(1);
    cfg.stream = st;
    return cudaLaunchKernelEx(&cfg, reset_kernel, head);        // this launch's error, not the runtime's last one
}

}  // namespace mmee

// The search kernel: every mapping decided, capacity pruning, top-k, in one launch.
//
// Work decomposition.  CTA c takes one tiling out of every `grid` consecutive ones, so that tilings that cannot fit at
// all (large tiles, neighbours in the index order) spread evenly, and keeps those that can in a compact list with their
// size and stationary-pair tables in shared memory.  How many of their rows fit is counted per tiling over all orders
// (count_rows).  A tiling's items, (class of C, order) of the fused mode and (order, mode) of the unfused ones, are evaluated by
// a warp, one lane each: the least key, exact in 64 bits, in closed form (mmee_classes.cuh).  The tilings with the least
// bounds come first, and those whose bound cannot enter the result any more are left out.  No candidate, row or threshold is
// kept per mapping, and nothing but the CTA's result leaves the SM.
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
// One optimum; the k best; one optimum of a chain of searches; one optimum for each of several array shapes.
constexpr int kModeSingle = 0, kModeMulti = 1, kModeChain = 2, kModeArrays = 3;

// Weights of the rows of two and of six orders (see count_rows).
__device__ const CountWeights kCountWeights[2] = {count_weights(2), count_weights(6)};

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

__device__ __forceinline__ void release_next_kernel() { asm volatile("griddepcontrol.launch_dependents;"); }
__device__ __forceinline__ void wait_previous_kernel() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// ------------------------------------------------------------------------------------------------
// shared memory
// ------------------------------------------------------------------------------------------------

struct Shared {
    // What lanes index with different indices (the constant bank would serialise them), copied from the plan.
    OrderInfo order[kMaxOrders];
    CountWeights weights;
    uint8_t done[kMaxChunk];        // tilings of the current pass that were evaluated first
    uint8_t list[kMaxChunk];        // ... that are evaluated after them (k = 1: an equal part for each warp)
    uint32_t divs[4][MMEE_MAX_DIVISORS];
    uint32_t cofactors[4][MMEE_MAX_DIVISORS];       // dimension / divisor
    uint32_t pe_rows, pe_cols;      // the array's logical shape
    uint32_t row_folds[4][MMEE_MAX_DIVISORS], col_folds[4][MMEE_MAX_DIVISORS];      // register-file tiling only
    alignas(16) longlong2 tops[kWarps][MMEE_MAX_TOPK];
    longlong2 up;                   // k > 1: nothing that follows this pair is among the k best
    long long kth[kWarps];          // finalize, k > 1: the k-th key of each warp's list (kInfKey: not full)
    unsigned long long feasible_rows[kWarps];
    uint32_t live_tilings[kWarps];
    uint32_t n_live;                // tilings of the current pass that can fit
    long long bound;                // chained searches: the bound that the search before left
    long long best;                 // ... the least key of a warp so far
    uint32_t n_list, cursor;        // k > 1: entries of `list`, next one to be taken
    uint32_t found;                 // chained searches, merging CTA: the search found something
    uint32_t count_cursor;          // next 32 units of the count
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

// k > 1: a pair that at least k of the entries of the warps' lists (sh.tops) do not follow; in all lanes.  If q warps hold r
// entries up to a pair each and q * r >= k, that is one: the least over four ways to cut k.
__device__ __forceinline__ void bound_of_lists(const Shared& sh, int k, int lane, int64_t& uk, uint64_t& ui) {
    static_assert(kWarps == 8, "eight lists, four cuts");
    const int most = kWarps >> (lane >> 3);                 // warps: 8, 4, 2, 1
    const int r = (k + most - 1) / most, q = (k + r - 1) / r;
    const longlong2 v = sh.tops[lane & 7][r - 1];
    int rank = 0;                                           // of this warp's r-th entry among those
#pragma unroll
    for (int j = 0; j < kWarps; ++j) {
        const int64_t ok = __shfl_sync(kFull, (int64_t)v.x, (lane & 24) + j);
        const uint64_t oi = __shfl_sync(kFull, (uint64_t)v.y, (lane & 24) + j);
        rank += pair_less(ok, oi, v.x, (uint64_t)v.y) || (ok == v.x && oi == (uint64_t)v.y && j < (lane & 7)) ? 1 : 0;
    }
    uk = rank == q - 1 ? v.x : kInfKey;
    ui = rank == q - 1 ? (uint64_t)v.y : UINT64_MAX;
    warp_min_pair(uk, ui);
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
__device__ __forceinline__ void load_shared(const Plan& p, uint32_t pe_rows, uint32_t pe_cols, Shared& sh) {
    const int tid = threadIdx.x;
    for (int i = tid; i < (int)(sizeof(sh.order) / 4); i += kSearchThreads)
        reinterpret_cast<uint32_t*>(sh.order)[i] = reinterpret_cast<const uint32_t*>(p.order)[i];
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

// The weights of the rows, by all threads of a CTA: those of the orders, on their way when this returns (await_weights), or one for
// every row that pruning keeps (PRUNED: where there may be such).
template <bool PRUNED>
__device__ __forceinline__ void start_weights(const Plan& p, Shared& sh) {
    constexpr int kWords = sizeof(CountWeights) / 4;
    if (PRUNED && p.row_pruning) {
        // (a warp's 32 weights are one 16-byte word of the parameters: lanes that read different words there wait for one another)
        const uint4* packed = reinterpret_cast<const uint4*>(p.kept_weights);
#pragma unroll
        for (int j = 0; j < (kWords + kSearchThreads - 1) / kSearchThreads; ++j) {
            const int i = (int)threadIdx.x + j * kSearchThreads;
            if (i >= kWords) break;
            const uint4 v = packed[i / 32];
            const uint32_t lo = i & 8 ? v.y : v.x, hi = i & 8 ? v.w : v.z;
            (&sh.weights.w[0][0][0])[i] = (i & 16 ? hi : lo) >> (4 * (i & 7)) & 15u;
        }
        return;
    }
    const int4* from = reinterpret_cast<const int4*>(&kCountWeights[p.n_orders == kMaxOrders ? 1 : 0]);
    int4* to = reinterpret_cast<int4*>(&sh.weights);
    for (int i = threadIdx.x; i < kWords / 4; i += kSearchThreads)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(to + i)), "l"(from + i) : "memory");
}
__device__ __forceinline__ void await_weights() { asm volatile("cp.async.wait_all;" ::: "memory"); }

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

// Waits for `n` CTAs to have published their parts, limited as above.
__device__ __forceinline__ bool await_parts(const SearchHeader* head, uint32_t n, uint32_t polls) {
#pragma unroll 4
    for (uint32_t i = 0; i < polls; ++i) {
        uint32_t now;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(now) : "l"(&head->done_ctas[0]) : "memory");
        if (now >= n) return true;
    }
    return false;
}
__device__ __forceinline__ void add_part(SearchHeader* head) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&head->done_ctas[0]) : "memory");
}

// Whether a chain's CTAs keep their tables from search to search.  They then count the rows that fit under a search's bound while
// they wait for its end, and add the count to its record before they publish their part of the next one.  Else, and in the
// launch's last search, the count is a part of what they publish.
__device__ __forceinline__ bool tables_stay(const Plan& p, const LaunchShape& shape) {
    return (uint64_t)shape.chunk * shape.grid >= p.t_end - p.t_begin;
}

// The end of a chained search, by all threads of one CTA; its record is made by another (resolve_chain).  True in warp 0: found.
// FRONT: the least (energy, latency, block) of all CTAs is the next point of the energy-latency front.  It is left as a
// latency optimum under that energy; the next search allows one word less of latency.
// Else: the least (energy, block, buffer need); the next search allows one word of buffer less than that need.
template <bool FRONT>
__device__ __forceinline__ bool finalize_chain(const Plan& p, int64_t cap_words, Shared& sh, ChainRecord* chain_to, uint32_t epoch, bool last,
                                               bool own_counts, SearchHeader* __restrict__ head, const Partial* __restrict__ partials, int n_partials) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int64_t ek = kInfKey, el = kInfKey;
    uint64_t ei = UINT64_MAX;
    unsigned long long rows = 0;
    for (int c0 = tid; c0 < n_partials; c0 += 2 * kSearchThreads) {
        longlong2 v[2], w[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int c = c0 + u * kSearchThreads;
            v[u] = make_longlong2(kInfKey, -1ll);
            w[u] = make_longlong2(-1ll, 0);
            if (c < n_partials) {
                v[u] = __ldcg(&partials[c].e[0]);
                w[u] = __ldcg(&partials[c].e[1]);
            }
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            rows += (unsigned long long)w[u].y;
            if (triple_less(v[u].x, v[u].y, (uint64_t)w[u].x, ek, el, ei)) { ek = v[u].x; el = v[u].y; ei = (uint64_t)w[u].x; }
        }
    }
    if (own_counts) {
        for (int off = 16; off; off >>= 1) rows += __shfl_down_sync(kFull, rows, off);
        if (lane == 0) sh.feasible_rows[warp] = rows;
    }
    warp_min_triple(ek, el, ei);
    if (lane == 0) {
        sh.tops[warp][0] = make_longlong2((long long)ek, (long long)el);
        sh.tops[warp][1] = make_longlong2((long long)ei, 0);
    }
    __syncthreads();
    if (warp) return false;
    ek = sh.tops[lane & (kWarps - 1)][0].x;
    el = sh.tops[lane & (kWarps - 1)][0].y;
    ei = (uint64_t)sh.tops[lane & (kWarps - 1)][1].x;
    warp_min_triple(ek, el, ei);
    const bool found = ek != kInfKey;
    if (lane == 0) {
        unsigned long long fit = 0;         // (the CTAs add theirs, else)
        if (own_counts)
            for (int w = 0; w < kWarps; ++w) fit += sh.feasible_rows[w];
        if (FRONT) *chain_to = {(long long)(found ? el : kInfKey), (unsigned long long)ei, fit, (long long)ek, 0, 0};
        else *chain_to = {(long long)ek, (unsigned long long)el, fit, (long long)cap_words, (long long)ei, 0};
        const int64_t bound = !found ? kNoBound : (FRONT ? el : (int64_t)ei) - 1;
        const unsigned long long word = (unsigned long long)epoch << 32 | (found ? (uint32_t)bound : 0xffffffffu);
        head->chain_bound = bound;
        if (!found || last) head->done_ctas[0] = 0;
        asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(&head->chain_epoch), "l"(word) : "memory");
    }
    return found;
}

// A CTA of its own merges the parts of a chain's searches: it does not have to count rows before it takes up the next one.
template <bool FRONT>
__device__ __noinline__ void merge_chain(const Plan& p, const LaunchShape& shape, Shared& sh, SearchHeader* head, const Partial* partials) {
    int64_t cap = shape.chain_read && !FRONT ? *reinterpret_cast<volatile long long*>(&head->chain_bound) : p.cap_words;
    const bool stay = tables_stay(p, shape);
    for (uint32_t step = 0; step < shape.chain_steps; ++step) {
        if (threadIdx.x == 0) sh.waited = await_parts(head, (step + 1) * shape.grid, shape.chain_polls) ? 1u : 0u;
        __syncthreads();
        if (!sh.waited) return;
        const bool found = finalize_chain<FRONT>(p, cap, sh, shape.chain_to + step, shape.chain_epoch + step, step + 1 == shape.chain_steps,
                                                 !stay || step + 1 == shape.chain_steps, head, partials, (int)shape.grid);
        if (threadIdx.x == 0) sh.found = found ? 1u : 0u;
        __syncthreads();
        if (!sh.found) return;
        if (!FRONT) cap = *reinterpret_cast<volatile long long*>(&head->chain_bound);
    }
}

// Run by every thread of ONE CTA (the last one to finish) after all CTAs have published their partial lists.
template <int OBJ, int MODE>
__device__ __noinline__ void finalize_step(const Plan& p, const LaunchShape& shape, const Limits& lim, Shared& sh, SearchHeader* __restrict__ head,
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
        wait_previous_kernel();                     // from here on the result records are touched
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
        wait_previous_kernel();
        const unsigned long long* from = reinterpret_cast<const unsigned long long*>(&best);
        unsigned long long* to = reinterpret_cast<unsigned long long*>(out_best);
        for (int i = lane; i < kWords; i += 32) to[i] = from[i];
    } else if (tid == 32) {
        // ready for the next search on this scratch
        unsigned long long all_live = 0;
        for (int w = 0; w < kWarps; ++w) all_live += sh.live_tilings[w];
        head->bound[shape.turn] = kInfKey;
        const uint32_t unfused_modes = (p.fuse_mask >> 1 & 1u) + (p.fuse_mask >> 2 & 1u);
        head->done_ctas[shape.turn] = 0;
        if (shape.stats) {
            wait_previous_kernel();         // (the searches before write them as well)
            shape.stats[0] = n_groups;
            shape.stats[1] = all_live * p.n_orders * ((p.fuse_mask & 1u ? kFusedReps : 0u) + (unfused_modes ? 18u : 0u));
        }
    }
}

// The full record of an optimum, by one CTA after load_shared: the first mapping with key `key` of block `where`.  key
// kInfKey: nothing fits.
// STAIRS: the first one that also has the buffer need `need`, the least of them.  A search that returns the first mapping
// with the least key and then searches on with one word less than that mapping's need would meet those with larger needs
// before it: the record's n_feasible is the number of mappings that fit under the last bound of such a sequence.  Where
// that is not the bound this one was found under, reserved2[0] says what it is, plus one (a rare case: index order
// raises needs), and the caller searches there.
// fitting(n): sets n to the number of mappings that fit (one thread); false: it did not come, and no record is written.
template <int OBJ, bool STAIRS, class Fitting>
__device__ __forceinline__ void resolve_record(const Plan& p, const Limits& lim, Shared& sh,
                                               int64_t key, uint64_t where, Fitting fitting, int64_t need, mmee_result_t* out) {
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
        bool came = true;
        if (lane == 0) {
            r.n_total = (p.t_end - p.t_begin) * (uint64_t)p.rows_per_tiling * 9u;
            unsigned long long n = 0;
            came = fitting(n);
            r.n_feasible = n;
            if (STAIRS) r.reserved2[0] = before_need;
        }
        if (!__shfl_sync(kFull, came ? 1 : 0, 0)) return;
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
    const bool stay = tables_stay(p, shape);
    for (uint32_t i = 0; i < shape.chain_steps; ++i) {
        __syncthreads();
        uint32_t low;
        if (threadIdx.x == 0) sh.waited = await_epoch(head, shape.chain_epoch + i, shape.chain_polls, low) ? 1u : 0u;
        __syncthreads();
        if (!sh.waited) return;
        const volatile ChainRecord* from = shape.chain_to + i;
        const ChainRecord c = {from->key, from->where, 0, from->bound, from->need, 0};
        const bool later = stay && c.key != kInfKey && i + 1 < shape.chain_steps;        // the count comes with the next search
        auto fitting = [&](unsigned long long& n) {
            uint32_t unused;
            if (later && !await_epoch(head, shape.chain_epoch + i + 1, shape.chain_polls, unused)) return false;
            n = from->n_feasible * p.n_sm;
            return true;
        };
        if (i % kRecordCtas == which) {
            if (FRONT) resolve_record<MMEE_OBJ_LATENCY_ECAP, false>(p, Limits{p.cap_words, c.bound}, sh, c.key, c.where, fitting, 0, out + i);
            else resolve_record<MMEE_OBJ_ENERGY, true>(p, Limits{c.bound, 0}, sh, c.key, c.where, fitting, c.need, out + i);
        }
        if (c.key == kInfKey) return;
    }
}

// ------------------------------------------------------------------------------------------------
// the search kernel
// ------------------------------------------------------------------------------------------------

// Searches launched one after the other overlap (programmatic dependent launch): the next one's CTAs move in as this one's
// leave, publish into a scratch of their own and merge, and only the records wait for the end of the search before, right before
// they are written, so that searches end in order.  A handle has kScratches scratches in turn.  Every (kScratches - 1)-th of its
// searches (`hold`) lets the next kernel start only after the kernel before it has ended (CTA 0 waits for that; the others need
// not): of two searches with the same scratch the second then starts after a search between them has seen the first one's end.
// (The turns of searches that a stream capture records count along: see search_on.)
// A kernel that is not launched this way follows a search as usual, and a search follows one as usual.  The waits are the
// hardware's grid dependency; a CTA waits for none that could start after it.

// Tells the host that what the CTA's threads have written is there.  All threads of the CTA.
__device__ __forceinline__ void signal_host(uint32_t* signal, uint32_t value) {
    if (!signal) return;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence_system();
        asm volatile("st.release.sys.global.u32 [%0], %1;" ::"l"(signal), "r"(value) : "memory");
    }
}

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
__device__ __forceinline__ void build_tile(const Plan& p, const Shared& sh, int sub, TileTab* tb) {
    uint32_t b[8];
#pragma unroll
    for (int d = 0; d < 8; ++d) b[d] = tb->b[d];
    if (TERMS && sub < 6) {
        const int op = sub >= 3 ? 1 : 0, sm = sub - 3 * op;
        int64_t P, Q;
        stationary_terms(p, SharedDivisors{sh}, b, op, sm, P, Q);
        (op ? tb->st.P2 : tb->st.P1)[sm] = P;
        (op ? tb->st.Q2 : tb->st.Q1)[sm] = Q;
    }
    for (int i = sub; i < kSizeSlots; i += 8) tb->size[i] = sat_size(size_words(p.dim, tb->b + 4, i));
}

template <int OBJ, int MODE>
__global__ void __launch_bounds__(kSearchThreads, 2)
search_kernel(const __grid_constant__ Plan p, const LaunchShape shape, SearchHeader* __restrict__ head, Partial* __restrict__ partials,
              mmee_result_t* __restrict__ out_best, mmee_result_t* __restrict__ out_topk) {
    constexpr bool SINGLE = MODE == kModeSingle, MULTI = MODE == kModeMulti, CHAIN = MODE == kModeChain, ARRAYS = MODE == kModeArrays;
    constexpr bool FRONT = CHAIN && OBJ == MMEE_OBJ_ENERGY_LCAP;      // least (energy, latency) under a bound on the latency
    constexpr bool STAIRS = CHAIN && OBJ == MMEE_OBJ_ENERGY;          // least (energy, block, buffer need) under a capacity
    static_assert(FRONT || STAIRS || !CHAIN, "only the searches of the Pareto fronts are chained");
    __shared__ Shared sh;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (!shape.hold) release_next_kernel();
    if (!CHAIN || blockIdx.x < shape.grid) start_weights<SINGLE>(p, sh);
    load_shared(p, p.pe_rows, p.pe_cols, sh);
    // Array shapes: the stationary-pair terms of shape y and tiling slot i at [y * chunk + i], behind the tilings' tables;
    // the warps' best items of shape y in sh.tops[.][y].
    StatTerms* terms = reinterpret_cast<StatTerms*>(&sh.tile[shape.chunk]);
    if (ARRAYS && tid < kWarps * (int)MMEE_MAX_TOPK) sh.tops[tid / (int)MMEE_MAX_TOPK][tid % (int)MMEE_MAX_TOPK] = make_longlong2(kInfKey, -1ll);
    static_assert(kMaxChunk <= 256 && kMaxChunk <= 32 * kWarps, "one byte per table, one lane per table");

    if (tid < (int)kMaxChunk) sh.done[tid] = 0;
    if (tid == 0) {
        sh.n_live = sh.n_list = sh.cursor = sh.count_cursor = 0;
        sh.check_failed = 0;
        sh.best = kInfKey;
    }
    __syncthreads();

    if (CHAIN && blockIdx.x >= shape.grid) {
        if (blockIdx.x < shape.grid + kRecordCtas) resolve_chain<FRONT>(p, shape, sh, head, blockIdx.x - shape.grid, out_topk);
        else merge_chain<FRONT>(p, shape, sh, head, partials);
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

    // A warp evaluates `per` tilings at a time, `n_items` lanes each: this lane the tiling `sub`, its fused block of order `os` with
    // C at class c, or its block of that order and unfused mode phi.
    const uint32_t fused_items = (p.fuse_mask & 1u) ? 3u * n_orders : 0u, unfused_modes = (p.fuse_mask >> 1 & 1u) + (p.fuse_mask >> 2 & 1u);
    const uint32_t n_items = fused_items + unfused_modes * n_orders;
    const uint32_t per = 32u / n_items, sub = (uint32_t)lane / n_items, item = (uint32_t)lane - sub * n_items;
    const bool fused = item < fused_items;
    const uint32_t mode = (fused ? item : item - fused_items) / n_orders, os = item % n_orders;     // class of C, or how many modes before phi
    const int c = fused ? (int)mode : 0, phi = fused ? 0 : (mode || !(p.fuse_mask & 2u) ? 2 : 1);
    const uint32_t block = os + (fused ? 0u : p.n_fused_blocks + mode * n_orders);
    const OrderInfo& oi = sh.order[os];

    // the best item so far: k = 1 of this thread, else the warp's list (lane j holds entry j)
    int64_t ek = kInfKey;
    uint64_t ei = UINT64_MAX;
    int64_t el = kInfKey;           // FRONT: its latency.  STAIRS: (el, ei) are the block and its need
    unsigned long long my_rows = 0;
    uint32_t my_live = 0;

    int64_t uk = kInfKey;           // nothing that follows this pair is among the k best
    uint64_t ui = UINT64_MAX;
    auto offer = [&](int64_t key, uint32_t id, bool valid) {
        if (!MULTI) {
            if (valid && pair_less(key, id, ek, ei)) { ek = key; ei = id; }
            return;
        }
        const int64_t lk = __shfl_sync(kFull, ek, k - 1);
        const uint64_t li = __shfl_sync(kFull, ei, k - 1);
        const bool pend = valid && key != kInfKey && pair_less(key, id, lk, li) && !pair_less(uk, ui, key, id);
        if (__any_sync(kFull, pend)) warp_offer(ek, ei, k, key, id, pend, lane);
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

    // The items of up to `per` tilings, this lane's of the one in table `slot` (`valid`: there is one; else any table) with the
    // stationary-pair terms `st`.
    auto evaluate_with = [&](uint32_t slot, bool valid, const StatTerms& st) {
        const TileTab& tb = sh.tile[slot];
        const uint32_t id = tb.t * p.n_blocks + block;
        int64_t x = kNoRow, x1 = 0, x2 = 0;
        int need = 0;
        if (fused_items) {
            const bool mine = valid && fused;
            fused_words<STAIRS>(tb, oi, dw, c, capc, [&](bool v) { return any(v && mine); }, x, need);
        }
        if (unfused_modes) {
            int need2;
            unfused_words<STAIRS>(tb, oi, dw, capc, x1, x2, need2);
            if (!fused) { x = x1; need = need2; }
        }
        const bool some = valid && x < kNoRow;
        if (!any(some)) return;
        const int64_t y = some ? x : 0, y1 = some ? x1 : 0, y2 = some ? x2 : 0, pass = phi == 2 ? 2 * dw.il : 0;
        const int64_t rho = fused && oi.recompute[c] != 0 ? (int64_t)tb.b[LOOP_J] : 1;
        auto key = [&]() {
            if (OBJ == MMEE_OBJ_ENERGY)         // (one form for both kinds)
                return fused_least_key<OBJ>(st, fused ? y : y1 + y2 + pass, rho, p.sm_mask, p.c_dram_gb, lim.key_cap);
            return fused ? fused_least_key<OBJ>(st, y, rho, p.sm_mask, p.c_dram_gb, lim.key_cap)
                         : unfused_least_key<OBJ>(st, y1, y2, pass, p.sm_mask, p.c_dram_gb, lim.key_cap);
        };
        if (FRONT) {
            // No mapping of the item is faster than this; after the first search few are fast enough (front of 10 816
            // tilings, one point: 53.9 us without this test, 52.5 with it).
            const int64_t q1 = min3(st.Q1), q2 = min3(st.Q2);
            const int64_t least = fused ? max64(y, q1 * rho + q2) : max64(y1, q1) + pass + max64(y2, q2);
            const bool can = some && least <= lim.key_cap;
            auto pair = [&](int s, int64_t& e, int64_t& l) {
                e = p.c_dram_gb * (fused ? y : y1 + y2 + pass) + st.P1[s / 3] * rho + st.P2[s % 3];
                l = fused ? max64(y, st.Q1[s / 3] * rho + st.Q2[s % 3]) : max64(y1, st.Q1[s / 3]) + pass + max64(y2, st.Q2[s % 3]);
            };
            if (any(can)) offer_front(pair, id, can);
        } else if (STAIRS) {
            offer_stairs(key(), id, need, some);
        } else {
            offer(key(), id, some);
        }
    };
    auto evaluate = [&](uint32_t slot, bool valid) { evaluate_with(slot, valid, sh.tile[slot].st); };

    // How many rows fit: units of one (A, B) of a tiling.  (Units of one (A, B, C) where those of a CTA fill no more than half of its
    // lanes: no gain, 768 tilings for k = 3 39.1 us and 38.9 without, tiny power-of-two tilings 7.15 and 7.14.  Code of their own for two
    // orders only where a single optimum is searched: it costs the others, which gain nothing, up to 2 % by its length alone.)
    auto count_fitting = [&](uint32_t n_tiles) {
        const uint32_t c0 = fused_items ? 0u : 4u, c1 = unfused_modes ? 5u : 4u, units = 9u * n_tiles;
        while (true) {
            uint32_t i = 0;
            if (lane == 0) i = atomicAdd(&sh.count_cursor, 32u);
            i = __shfl_sync(kFull, i, 0);
            if (i >= units) break;
            i += (uint32_t)lane;
            const bool valid = i < units;
            const uint32_t ab = valid ? i / n_tiles : 0u;
            const uint32_t n = count_rows(sh.tile[valid ? i - ab * n_tiles : 0u].size, (int)ab, (int)c0, (int)c1,
                                          SINGLE && p.row_pruning ? 1u : unfused_modes, capc, sh.weights, SINGLE && n_orders == 2u, [&](bool v) { return any(v && valid); });
            if (valid) my_rows += n;
        }
    };

    const bool one_pass = CHAIN && tables_stay(p, shape);
    // chained: the best triple of this lane's tiling (see below), the tiling's first block and the least that it has of what is
    // bounded (latency, buffer need)
    int64_t ck = kInfKey, cl = 0;
    uint64_t ci = 0, first = 0;
    int64_t limited = 0;
    bool valid = false;
    for (uint32_t step = 0;; ++step) {
        // chained: the rows that fit under the bound before; whether those of this one are counted before it is published, or the
        // count of the launch's first search stands (the bound is on the latency)
        const bool last = CHAIN && step + 1 == shape.chain_steps, counted = FRONT && one_pass && step;
        const bool count_now = !counted && (!one_pass || last);
        if (CHAIN && !counted) my_rows = 0;
        int64_t bk = kInfKey, bl = kInfKey;       // chained: the warp's best triple
        uint64_t bi = UINT64_MAX;
        if (CHAIN && (step || shape.chain_read)) {
            __syncthreads();                // the counters of the search before are no longer in use
            if (tid == 0) {
                uint32_t low = 0;
                const bool over = !step || await_epoch(head, shape.chain_epoch + step - 1, shape.chain_polls, low);
                if (!over) sh.bound = kNoBound;
                else if (step && STAIRS) sh.bound = low == 0xffffffffu ? kNoBound : (int64_t)low;
                else sh.bound = *reinterpret_cast<volatile long long*>(&head->chain_bound);
                sh.count_cursor = 0;
                sh.best = kInfKey;
                if (!one_pass) sh.n_live = 0;
            }
            __syncthreads();
            const int64_t bound = sh.bound;
            if (bound == kNoBound) return;
            if (tid == 0 && step && one_pass) {     // (before this thread says that the CTA's next part is there)
                unsigned long long rows = 0;
                for (int w = 0; w < kWarps; ++w) rows += sh.feasible_rows[w];
                atomicAdd(&shape.chain_to[step - 1].n_feasible, rows);
            }
            if (STAIRS) {
                lim.cap_words = bound;
                capc = (int)bound;
            } else {
                lim.key_cap = bound;
            }
        }
        // Tiling number m of this CTA is one of the m-th `grid` consecutive ones, a different one in every round (a fixed
        // one would be the same divisor of the last dimension again and again).
        for (uint32_t m0 = 0; (uint64_t)m0 * grid < n_tilings; m0 += shape.chunk) {
            if (m0) {
                __syncthreads();                // the previous pass's tables are no longer in use
                if (tid == 0) sh.n_live = sh.n_list = sh.cursor = sh.count_cursor = 0;
                if (tid < (int)kMaxChunk) sh.done[tid] = 0;
                __syncthreads();
            }
            if (!step || !one_pass) {
                // the tilings that can fit, one per thread: with every operand at L3 the buffer need is smallest,
                // max(A+B+C, C+D+E) tiles (Eq. 1-4)
                const uint32_t m = m0 + (uint32_t)tid;
                uint64_t rel = (uint64_t)m * grid + (blockIdx.x + m) % grid;
                uint32_t b[8], t = 0;
                bool live = (uint32_t)tid < shape.chunk && (uint64_t)m * grid < n_tilings && rel < n_tilings;
                if (live) {
                    t = (uint32_t)(p.t_begin + rel);
                    tiling_bounds(p, SharedDivisors{sh}, t, b);
                    const uint64_t ta = (uint64_t)b[4] * b[5], tbb = (uint64_t)b[5] * b[6], tc = (uint64_t)b[4] * b[6];
                    const uint64_t td = (uint64_t)b[6] * b[7], te = (uint64_t)b[4] * b[7];
                    live = ta + tbb + tc <= (uint64_t)capc && tc + td + te <= (uint64_t)capc;
                }
                const unsigned who = __ballot_sync(kFull, live);
                uint32_t at = 0;
                if (who && lane == 0) at = atomicAdd(&sh.n_live, (uint32_t)__popc(who));
                at = __shfl_sync(kFull, at, 0) + (uint32_t)__popc(who & ((1u << lane) - 1u));
                if (live) {
                    TileTab& tb = sh.tile[at];
                    tb.t = t;
#pragma unroll
                    for (int d = 0; d < 8; ++d) tb.b[d] = b[d];
                }
                __syncthreads();
                // their tables, eight threads each
                const uint32_t n_live = sh.n_live;
                for (uint32_t i = (uint32_t)tid; i - (uint32_t)lane < 8u * n_live; i += kSearchThreads) {
                    const bool valid = i < 8u * n_live;
                    TileTab& tb = sh.tile[valid ? i / 8u : 0u];
                    if (valid) build_tile<!ARRAYS>(p, sh, (int)(i & 7u), &tb);
                    if (!ARRAYS && !CHAIN) {
                        __syncwarp();
                        if (valid && (i & 7u) == 7u) tb.least = tile_least_key<OBJ>(tb.st, dw, p.c_dram_gb, lim.key_cap);
                    }
                }
            }
            if (!step && !m0) await_weights();
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

            const uint32_t n_tiles = sh.n_live;
            if (tid == 0) my_live += n_tiles;

            // ---- the least keys: first of the tilings whose bound (tile_least_key) is smallest among a warp's own, by half of the warps for a single
            // optimum (the others count meanwhile), by all for the k best
            const bool all_at_once = ARRAYS || CHAIN || n_tiles <= per * (uint32_t)kWarps;
            if (CHAIN) {
                // This lane keeps the best triple of its tiling over the searches: valid while it is within the bound, else a triple
                // that the tiling's best one does not precede.  The warp evaluates the most promising of those until its best
                // triple is a valid one, or worse than another warp's.  (Front of the GPT-3 FFN, evaluating every tiling that
                // fits in each of its twenty searches: 242 us.)
                const uint32_t own = (uint32_t)(warp + kWarps * lane);
                if (!step || !one_pass) {
                    valid = false;
                    ck = kInfKey;
                    if (own < n_tiles) {
                        const TileTab& tb = sh.tile[own];
                        ck = tile_least_key<OBJ>(tb.st, dw, p.c_dram_gb, INT64_MAX);
                        first = (uint64_t)tb.t * p.n_blocks;
                        const int one = sat_add(tb.size[S_ik], tb.size[S_kl]), two = sat_add(tb.size[S_lj], tb.size[S_ij]);
                        limited = FRONT ? tile_least_key<MMEE_OBJ_LATENCY>(tb.st, dw, 0, 0) : (int64_t)sat_add(tb.size[S_il], one > two ? one : two);
                    }
                }
                if (valid && (FRONT ? cl > lim.key_cap : (int64_t)ci > lim.cap_words)) valid = false;
                if (limited > (FRONT ? lim.key_cap : lim.cap_words)) ck = kInfKey;
                while (true) {
                    int64_t mk = ck, ml = valid ? cl : (STAIRS ? (int64_t)first : 0);
                    uint64_t mi = valid ? ci : 0;
                    const int64_t own_l = ml;
                    const uint64_t own_i = mi;
                    warp_min_triple(mk, ml, mi);
                    if (mk == kInfKey || mk > *reinterpret_cast<volatile long long*>(&sh.best)) break;
                    const unsigned who = __ballot_sync(kFull, ck == mk && own_l == ml && own_i == mi);
                    if ((__ballot_sync(kFull, valid) >> (__ffs(who) - 1)) & 1u) {
                        if (lane == 0) atomicMin(&sh.best, (long long)mk);
                        if (triple_less(mk, ml, mi, bk, bl, bi)) { bk = mk; bl = ml; bi = mi; }
                        break;
                    }
                    // up to `per` tilings
                    uint32_t slot = 0;
                    int src = 0;
                    bool chosen = false;
                    uint32_t n = 0;
#pragma unroll 1
                    for (; n < per; ++n) {
                        int at = __ffs(who) - 1;
                        if (n) {
                            int64_t lk = valid || chosen ? kInfKey : ck;
                            uint64_t li = valid || chosen ? UINT64_MAX : first;
                            const uint64_t own_first = li;
                            warp_min_pair(lk, li);
                            if (lk == kInfKey) break;
                            at = __ffs(__ballot_sync(kFull, own_first == li)) - 1;
                        }
                        if (lane == at) chosen = true;
                        if (sub >= n) slot = (uint32_t)(warp + kWarps * at);
                        if (sub == n) src = at;
                    }
                    ek = el = kInfKey;
                    ei = UINT64_MAX;
                    evaluate(slot, sub < n);
#pragma unroll 1
                    for (uint32_t j = 0; j < n; ++j) {
                        int64_t tk = sub == j ? ek : kInfKey, tl = sub == j ? el : kInfKey;
                        uint64_t ti = sub == j ? ei : UINT64_MAX;
                        warp_min_triple(tk, tl, ti);
                        const int at = __shfl_sync(kFull, src, (int)(j * n_items));
                        if (lane == at) { ck = tk; cl = tl; ci = ti; valid = tk != kInfKey; }
                    }
                }
            } else if (ARRAYS) {
                // One shape and up to 32 tilings by a warp, fewer where there are fewer shapes than warps: those whose least key may
                // still be better, the most promising first, `per` at a time.
                // (Two orders, seven shapes, 8 820 tilings: 45.6 us with one tiling at a time, 39.7 so; one shape, 72 tilings, eight
                // to a CTA: 32.3 us with one warp for the shape, 28.1 with as many as its tilings fill, which leaves the others to count.)
                const uint32_t parts = max((n_tiles + 31u) / 32u, min((uint32_t)kWarps / shape.n_arrays, (n_tiles + per - 1u) / per));
                for (uint32_t u = (uint32_t)warp; u < shape.n_arrays * parts; u += kWarps) {
                    const uint32_t y = u / parts, part = u - y * parts, mine = part + parts * (uint32_t)lane;
                    const longlong2 own = sh.tops[warp][y];
                    ek = own.x;
                    ei = (uint64_t)own.y;
                    const StatTerms* st = terms + y * shape.chunk;
                    bool open = mine < n_tiles;
                    const uint64_t first = open ? (uint64_t)sh.tile[mine].t * p.n_blocks : UINT64_MAX;
                    const int64_t least = open ? tile_least_key<OBJ>(st[mine], dw, p.c_dram_gb, lim.key_cap) : kInfKey;
                    while (true) {
                        int64_t bk = ek;
                        uint64_t bi = ei;
                        warp_min_pair(bk, bi);
                        uint32_t slot = 0, n = 0;
                        for (; n < per; ++n) {
                            int64_t lk = open ? least : kInfKey;
                            uint64_t li = open ? first : UINT64_MAX;
                            warp_min_pair(lk, li);
                            if (!pair_less(lk, li, bk, bi)) break;
                            const unsigned who = __ballot_sync(kFull, open && first == li);
                            const int src = __ffs(who) - 1;
                            if (lane == src) open = false;
                            if (sub >= n) slot = part + parts * (uint32_t)src;
                        }
                        if (!n) break;
                        evaluate_with(slot, sub < n, st[slot]);
                    }
                    warp_min_pair(ek, ei);
                    if (lane == 0) sh.tops[warp][y] = make_longlong2((long long)ek, (long long)ei);
                }
            } else if (all_at_once) {
                for (uint32_t i = (uint32_t)warp * per; i < n_tiles; i += per * (uint32_t)kWarps)
                    evaluate(i + sub < n_tiles ? i + sub : i, sub < per && i + sub < n_tiles);
            } else if (!m0 && (MULTI || warp < kWarps / 2)) {
                // (by the bound as a float, then by the index: where many bounds are the same, as those of the latency often are, the
                // lowest index is the best; which come first changes no result)
                const uint32_t every = MULTI ? (uint32_t)kWarps : (uint32_t)kWarps / 2u, own = (uint32_t)warp + (uint32_t)lane * every;
                uint32_t rank = 0xffffffffu, number = 0xffffffffu;
                if (own < n_tiles) {
                    rank = __float_as_uint(__ll2float_rn(sh.tile[own].least));
                    number = sh.tile[own].t << 5 | (uint32_t)lane;
                }
                uint32_t slot = 0;
                bool valid = false;
                for (uint32_t i = 0; i < per; ++i) {
                    const uint32_t least = __reduce_min_sync(kFull, rank);
                    const uint32_t first = __reduce_min_sync(kFull, rank == least ? number : 0xffffffffu);
                    if (least == 0xffffffffu) break;
                    const uint32_t src = first & 31u;
                    if ((uint32_t)lane == src) {
                        rank = 0xffffffffu;
                        sh.done[own] = 1;
                    }
                    if (sub >= i) slot = (uint32_t)warp + src * every;
                    if (sub == i) valid = true;
                }
                evaluate(slot, valid);
            }

            if (MULTI && !all_at_once) {
                // a bound for this CTA from the warps' lists, and for all CTAs
                if (lane < kTopK) sh.tops[warp][lane] = make_longlong2((long long)ek, (long long)ei);
                __syncthreads();
                if (!warp) {
                    bound_of_lists(sh, k, lane, uk, ui);
                    if (lane == 0 && uk != kInfKey) atomicMin(&head->bound[shape.turn], (long long)uk);
                }
            }

            if (!CHAIN || count_now) count_fitting(n_tiles);

            if (all_at_once) continue;
            // ---- what those left may be better than: nothing that follows it is among the k best
            if (MULTI) {
                if (tid == 0) {
                    const long long g = *reinterpret_cast<volatile long long*>(&head->bound[shape.turn]);
                    sh.up = g < uk ? make_longlong2(g, -1ll) : make_longlong2((long long)uk, (long long)ui);
                }
                __syncthreads();
                uk = sh.up.x;
                ui = (uint64_t)sh.up.y;
            } else {
                int64_t lk = ek;
                uint64_t li = ei;
                warp_min_pair(lk, li);
                // (not where the warp's result goes: another warp may be there before this one has read)
                if (lane == 0) sh.tops[warp][1] = make_longlong2((long long)lk, (long long)li);
                __syncthreads();
                const longlong2 v = sh.tops[lane & (kWarps - 1)][1];
                uk = v.x;
                ui = (uint64_t)v.y;
                warp_min_pair(uk, ui);
            }
            auto open = [&](uint32_t slot) {
                const TileTab& tb = sh.tile[slot];
                return !sh.done[slot] && tb.least != kInfKey && !pair_less(uk, ui, tb.least, (uint64_t)tb.t * p.n_blocks);
            };
            if (!MULTI) {
                // Every warp goes over all tilings and keeps each kWarps-th of those left: no barrier, and a warp's last evaluation
                // is seldom later than with one list for all (pruned sweep 10.1 us with that, 9.8 so; BERT 8.65 and 8.45).
                uint8_t* list = sh.list + warp * (int)(kMaxChunk / kWarps);
                static_assert(kMaxChunk % kWarps == 0, "equal parts");
                uint32_t n = 0;
                for (uint32_t at = 0; at < n_tiles; at += 32u) {
                    const uint32_t slot = at + (uint32_t)lane;
                    const bool left = slot < n_tiles && open(slot);
                    const unsigned m = __ballot_sync(kFull, left);
                    const uint32_t rank = n + (uint32_t)__popc(m & ((1u << lane) - 1u));
                    if (left && rank % kWarps == (uint32_t)warp) list[rank / kWarps] = (uint8_t)slot;
                    n += (uint32_t)__popc(m);
                }
                __syncwarp();
                const uint32_t n_mine = (n + (uint32_t)(kWarps - 1 - warp)) / kWarps;
                for (uint32_t i = 0; i < n_mine; i += per) evaluate(list[i + sub < n_mine ? i + sub : i], sub < per && i + sub < n_mine);
                continue;
            }
            // (k > 1: what a warp takes depends on how much better its own list has got.  Convolution chain top-16: 30.4 us, with
            // equal parts as above 31.0)
            {
                const uint32_t own = (uint32_t)(warp + kWarps * lane);
                bool left = own < n_tiles;
                const uint32_t own_slot = left ? own : 0u;
                left = left && open(own_slot);
                const unsigned m = __ballot_sync(kFull, left);
                uint32_t at = 0;
                if (m && lane == 0) at = atomicAdd(&sh.n_list, (uint32_t)__popc(m));
                at = __shfl_sync(kFull, at, 0) + (uint32_t)__popc(m & ((1u << lane) - 1u));
                if (left) sh.list[at] = (uint8_t)own_slot;
            }
            __syncthreads();
            const uint32_t n_list = sh.n_list;
            while (true) {
                uint32_t i = 0;
                if (lane == 0) i = atomicAdd(&sh.cursor, per);
                i = __shfl_sync(kFull, i, 0);
                if (i >= n_list) break;
                const uint32_t slot = sh.list[i + sub < n_list ? i + sub : i];
                // (the warp's own list may have got better)
                const int64_t lk = __shfl_sync(kFull, ek, k - 1);
                const uint64_t li = __shfl_sync(kFull, ei, k - 1);
                bool valid = sub < per && i + sub < n_list;
                valid = valid && pair_less(sh.tile[slot].least, (uint64_t)sh.tile[slot].t * p.n_blocks, lk, li);
                if (!any(valid)) continue;
                evaluate(slot, valid);
            }
        }

        // ---- this CTA's result
        unsigned long long rows_here = 0;
        if (!CHAIN || count_now || (counted && last)) {
            rows_here = my_rows;
            for (int off = 16; off; off >>= 1) rows_here += __shfl_down_sync(kFull, rows_here, off);
        }
        if (!CHAIN && lane == 0) sh.feasible_rows[warp] = rows_here;
        if (MULTI) {
            merge_warps(sh, k, lane, warp, ek, ei);
        } else if (CHAIN) {
            if (lane == 0) {
                sh.tops[warp][0] = make_longlong2((long long)bk, (long long)bl);
                sh.tops[warp][1] = make_longlong2((long long)bi, (long long)rows_here);
            }
            __syncthreads();
        } else if (!ARRAYS) {
            warp_min_pair(ek, ei);
            if (lane == 0) sh.tops[warp][0] = make_longlong2((long long)ek, (long long)ei);
            __syncthreads();
        }
        if (ARRAYS) {
            wait_previous_kernel();             // from here on the scratch is touched
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
                count = (uint32_t)__popc(__ballot_sync(kFull, ek != kInfKey));
                if (lane < (int)max(count, 1u)) out->e[lane] = make_longlong2((long long)ek, (long long)ei);
            } else if (CHAIN) {
                ek = sh.tops[lane & (kWarps - 1)][0].x;
                el = sh.tops[lane & (kWarps - 1)][0].y;
                ei = (uint64_t)sh.tops[lane & (kWarps - 1)][1].x;
                warp_min_triple(ek, el, ei);
                unsigned long long own = lane < kWarps ? (unsigned long long)sh.tops[lane][1].y : 0;
                for (int off = kWarps / 2; off; off >>= 1) own += __shfl_xor_sync(kFull, own, off);
                own = __shfl_sync(kFull, own, 0);
                count = 2;
                if (lane < 2) out->e[lane] = lane ? make_longlong2((long long)ei, (long long)own) : make_longlong2((long long)ek, (long long)el);
            } else {
                const longlong2 v = sh.tops[lane & (kWarps - 1)][0];
                ek = v.x;
                ei = (uint64_t)v.y;
                warp_min_pair(ek, ei);
                count = ek != kInfKey ? 1u : 0u;
                if (lane == 0) out->e[0] = make_longlong2((long long)ek, (long long)ei);
            }
            unsigned long long rows = !CHAIN && lane < kWarps ? sh.feasible_rows[lane] : 0;
            if (!CHAIN)
                for (int off = kWarps / 2; off; off >>= 1) rows += __shfl_down_sync(kFull, rows, off);
            if (!CHAIN && lane == 0) {
                out->count = count;
                out->live_tilings = my_live;
                out->feasible_rows = rows;
            }
            // Grid reduction without a wait: every CTA makes its partial list visible, then draws a ticket; the CTA that
            // draws the last one knows that all lists are there and runs the finalize step.
            __syncwarp();
            if (lane == 0) {
                if (CHAIN) add_part(head);
                else sh.last_cta = draw_ticket(&head->done_ctas[shape.turn]) == grid - 1 ? 1u : 0u;
            }
        }
        if (CHAIN) {
            if (last) return;
            if (one_pass && !counted) count_fitting(sh.n_live);
            if (one_pass) {
                rows_here = my_rows;
                for (int off = 16; off; off >>= 1) rows_here += __shfl_down_sync(kFull, rows_here, off);
                if (lane == 0) sh.feasible_rows[warp] = rows_here;
            }
            continue;
        }
        __syncthreads();
        if (shape.hold && (sh.last_cta || !blockIdx.x)) {
            if (!blockIdx.x) wait_previous_kernel();
            release_next_kernel();              // (takes effect once every CTA has said so or ended)
        }
        if (sh.last_cta) {
            finalize_step<OBJ, MODE>(p, shape, lim, sh, head, partials, (int)grid, out_best, out_topk);
            signal_host(shape.signal, shape.signal_value);
        }
        return;
    }
}

__global__ void reset_kernel(SearchHeader* head) {
    for (int i = 0; i < kScratches; ++i) {
        head->bound[i] = kInfKey;
        head->done_ctas[i] = 0;
    }
    head->chain_epoch = 0;
}

// Merge of the CTAs' best items of array shape blockIdx.x, and the record of the optimum.
template <int OBJ>
__global__ void __launch_bounds__(kSearchThreads, 2)
resolve_arrays_kernel(const __grid_constant__ Plan p, const LaunchShape shape, const Partial* partials, mmee_result_t* out) {
    __shared__ Shared sh;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    load_shared(p, shape.array[blockIdx.x][0], shape.array[blockIdx.x][1], sh);
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
    auto fitting = [&](unsigned long long& n) {
        n = rows * p.n_sm;
        return true;
    };
    resolve_record<OBJ, false>(p, Limits{p.cap_words, p.key_cap}, sh, ek, ei, fitting, 0, out + blockIdx.x);
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
                   : p.topk > 1    ? search_kernel<OBJ, kModeMulti> : search_kernel<OBJ, kModeSingle>;
    if (!kernel) return cudaErrorInvalidValue;
    const uint32_t grid = shape.chain_steps ? shape.grid + kChainExtraCtas : shape.grid;
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

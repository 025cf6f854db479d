// The search's evaluation of a whole block of mappings at once.
//
// A block is one (tiling, fusion mode, order): 3125 rows of buffering levels (625 unfused) times nine stationary pairs.
// What the search needs of it is exact but small: how many of its rows fit the buffer (Eq. 4), and its least key.
//
//   * Rows with equal class combinations (OrderInfo) have equal buffer needs and equal DRAM words, so that a fused
//     block holds 3*3*3*4*4 = 432 different rows of 3125, each standing for the product of its classes' widths.  The
//     two nests of an unfused block are independent: 9 + 9 different (A, B) and (D, E) choices of 625 rows.
//   * Every key is non-decreasing in the DRAM words at a fixed stationary pair and recompute flag (energy is a sum,
//     latency a maximum or a sum of maxima, their product monotone in both).  The least key of a block is therefore the
//     least, over stationary pairs, of the key at the LEAST DRAM words of the rows that fit: one 64-bit minimum per
//     (class of C), and nine keys at the end, instead of nine keys per row.
//   * For that minimum D and E have two candidates each, not four: left at L3 (no space while the other operator runs)
//     or held at the smallest class that is fetched once; every other class needs more space for the same words.
//
// Host and device: the functions are plain arithmetic on a size table, so that they can be checked on the CPU as well.
#pragma once

#include "mmee_plan.h"

namespace mmee {

constexpr int kSizeCap = (1 << 30) - 1;        // buffer sizes saturate here, above every admissible capacity
constexpr int64_t kNoRow = INT64_C(1) << 62;   // DRAM words of "no row fits"; sums of words stay below 2^62

// Stationary-pair terms of one tiling, linear in the recomputation factor rho of C (j_D or 1): energy P1[sm1] * rho + P2[sm2]
// (buffer<->PE words, MACs, softmax), compute words Q1[sm1] * rho + Q2[sm2].
struct StatTerms {
    int64_t P1[3], P2[3], Q1[3], Q2[3];
};

// What a CTA keeps of one tiling, shared by its orders and classes.
struct TileTab {
    int32_t  size[kSizeSlots];      // buffer words, saturated to kSizeCap
    uint32_t t;                     // tiling index
    uint32_t b[8];                  // bounds i_D, k_D, l_D, j_D, i_G, k_G, l_G, j_G
    StatTerms st;
    int64_t  least;                 // no mapping's key is smaller (tile_least_key)
};
static_assert(sizeof(TileTab) % 16 == 8, "lanes that read the same word of consecutive tables meet in pairs at most on a bank");

// Whole operands, the same for every tiling.
struct DimWords { int64_t ik, kl, lj, ij, il; };

MMEE_HD int sat_size(uint64_t v) { return v < (uint64_t)kSizeCap ? (int)v : kSizeCap; }
MMEE_HD int sat_add(int a, int b) { const int s = a + b; return s < kSizeCap ? s : kSizeCap; }
MMEE_HD int64_t min64(int64_t a, int64_t b) { return a < b ? a : b; }
MMEE_HD int64_t max64(int64_t a, int64_t b) { return a > b ? a : b; }

// Words of size slot `slot` of a tiling with tile extents g.  Six bits a slot: the two dimensions (bits 0-1, 2-3) and which
// of them is whole (bits 4, 5); ten slots to a word, so that lanes with different slots look nothing up.
constexpr uint64_t size_codes(int first) {
    constexpr uint8_t code[kSizeSlots] = {
        0x04, 0x24, 0x34, 0x09, 0x19, 0x39, 0x08, 0x18, 0x28, 0x38, 0x0e, 0x1e, 0x2e, 0x3e, 0x0c, 0x1c, 0x2c, 0x3c};
    uint64_t w = 0;
    for (int i = first; i < first + 10 && i < kSizeSlots; ++i) w |= (uint64_t)code[i] << (6 * (i - first));
    return w;
}
MMEE_HD uint64_t size_words(const uint32_t dim[4], const uint32_t g[4], int slot) {
    constexpr uint64_t lo = size_codes(0), hi = size_codes(10);
    const uint32_t c = (uint32_t)(slot < 10 ? lo >> (6 * slot) : hi >> (6 * (slot - 10)));
    const uint32_t x = c & 3u, y = (c >> 2) & 3u;
    return (uint64_t)((c & 16u) ? dim[x] : g[x]) * ((c & 32u) ? dim[y] : g[y]);
}

// ------------------------------------------------------------------------------------------------
// How many rows of a tiling fit, over all its blocks
// ------------------------------------------------------------------------------------------------
// What decides whether a row fits is the sizes of its five operands, and over all orders there are few different ones: three of
// A and of B, four of C, D and E each (SizeSlot), D and E also at L3, where they take no room while the other operator runs.
// Rows of all orders with the same sizes are counted together, by a weight that depends on the orders alone: 9 * 4 * 25
// comparisons decide a tiling's fused rows, where its blocks one by one need 6 * 3 * (4 * 9 + 5 * 16), and 9 * 16 more the
// unfused ones.
// (GQA latency, 14 336 tilings, one search after the other: 12.1 us with the counts of each block's classes, 10.1 so.)
struct alignas(16) CountWeights {
    uint32_t w[9][5][kCountChoices];           // [3 * class of A + class of B][size slot of C - S_il; 4: the rows of one unfused mode]
};
// The weights of the first n_orders orders (outer -> inner: I L J, L I J, I J L, L J I, J I L, J L I): products of the numbers of
// levels in the classes (OrderInfo::width).  In the nests of an unfused mode D and E at L3 are like their first retained class.
constexpr CountWeights count_weights(int n_orders) {
    CountWeights t = {};
    constexpr int level[6][3] = {{4, 3, 2}, {3, 4, 2}, {4, 2, 3}, {2, 4, 3}, {3, 2, 4}, {2, 3, 4}};     // beta - 3 of i2, l2, j2
    for (int o = 0; o < n_orders; ++o) {
        const int i = level[o][0], l = level[o][1], j = level[o][2];
        const int il0 = i < l ? i : l, il1 = i < l ? l : i, lj0 = l < j ? l : j, lj1 = l < j ? j : l, ij0 = i < j ? i : j, ij1 = i < j ? j : i;
        const int a[3] = {1, i - 1, 5 - i}, b[3] = {1, l - 1, 5 - l}, c[3] = {il0, il1 - il0, 5 - il1};
        const int d[4] = {1, lj0 - 1, lj1 - lj0, 5 - lj1}, e[4] = {1, ij0 - 1, ij1 - ij0, 5 - ij1};
        const int cs[3] = {0, i < l ? 1 : 2, 3}, d_lo = l < j ? 1 : 2, e_lo = i < j ? 1 : 2;
        for (int ab = 0; ab < 9; ++ab)
            for (int de = 0; de < 16; ++de) {
                const int x = de / 4, y = de % 4, n = a[ab / 3] * b[ab % 3] * d[x] * e[y];
                for (int k = 0; k < 3; ++k) t.w[ab][cs[k]][de_choice(x, y, d_lo, e_lo)] += (uint32_t)(n * c[k]);
                t.w[ab][4][de_choice(x ? x : 1, y ? y : 1, d_lo, e_lo)] += (uint32_t)n;
            }
    }
    return t;
}
// The rows that fit with A and B of class ab / 3, ab % 3 and choices c0 .. c1 - 1 of C (see CountWeights; those of choice 4
// `unfused` times).  ANY(x): true if x holds for some lane of the warp (device), for this call (host).
// TWO: of two orders, both with j2 innermost, whose rows have no D or E of the second of the four sizes: 16 choices of D and E
// instead of 25, 9 of 16 in the unfused modes.  (12 480 tilings, fused, one search after the other: 9.45 us with all, 9.1 so; 18 432
// tilings of all modes 11.3 and 10.8.)
template <bool TWO, class Any>
MMEE_HD uint32_t count_rows_of(const int32_t* size, int ab, int c0, int c1, uint32_t unfused, int capc, const CountWeights& w, Any any) {
    const int a = ab / 3, b = ab - 3 * a;
    const int A = size[S_ik + a], B = size[S_kl + b], AB = sat_add(A, B);
    int D[4], E[4];
#pragma unroll
    for (int x = 0; x < 4; ++x) {
        D[x] = size[S_lj + x];
        E[x] = size[S_ij + x];
    }
    // Room beside A, B, C: s while Op1 runs; s + more while Op2 runs, since A and B at L3 take none then.  What D or E at L3
    // need while Op2 runs, beyond that, is compared with s as well.  (Unfused: the room beside C, if A and B fit it.)
    const int more = sat_add(a ? 0 : A, b ? 0 : B);
    const int d3 = D[0] > more ? D[0] - more : 0, e3 = E[0] > more ? E[0] - more : 0, both3 = D[0] + E[0] > more ? D[0] + E[0] - more : 0;
    uint32_t n = 0;
#pragma unroll 1
    for (int c = c0; c < c1; ++c) {
        int s = capc - (c < 4 ? sat_add(AB, size[S_il + c]) : size[S_il]);
        if (c == 4 && AB > s) s = -1;
        if (!any(both3 <= s)) continue;         // (the least of all sums)
        const uint4* u = reinterpret_cast<const uint4*>(w.w[ab][c]);
        const int room[4] = {s - E[0], s - E[1], s - E[2], s - E[3]};
        uint32_t m = 0;
        auto add = [&](bool b0, bool b1, bool b2, bool b3, uint4 v) {
            if (b0) m += v.x;
            if (b1) m += v.y;
            if (b2) m += v.z;
            if (b3) m += v.w;
        };
#pragma unroll
        for (int x = 0; x < 4; ++x)
            if (!TWO || x != 1) add(D[x] <= room[0], !TWO && D[x] <= room[1], D[x] <= room[2], D[x] <= room[3], u[x]);
        if (c < 4) {
            add(D[0] <= s - e3, !TWO && D[1] <= s - e3, D[2] <= s - e3, D[3] <= s - e3, u[4]);
            add(d3 <= room[0], !TWO && d3 <= room[1], d3 <= room[2], d3 <= room[3], u[5]);
            m += both3 <= s ? w.w[ab][c][24] : 0u;
        } else {
            m *= unfused;
        }
        n += m;
    }
    return n;
}

template <class Any>
MMEE_HD uint32_t count_rows(const int32_t* size, int ab, int c0, int c1, uint32_t unfused, int capc, const CountWeights& w, bool two, Any any) {
    return two ? count_rows_of<true>(size, ab, c0, c1, unfused, capc, w, any) : count_rows_of<false>(size, ab, c0, c1, unfused, capc, w, any);
}

// ------------------------------------------------------------------------------------------------
// The least DRAM words of a block's rows that fit
// ------------------------------------------------------------------------------------------------
// Of an operand's classes two matter, three of A or B where C is regenerated: left at L3, which takes the least room, and the
// smallest class that is fetched once; the other classes take more room for the same words.  Only with j2 outermost and C
// regenerated the operand of the loop in the middle (A or B) has one more in between: class 1, fetched once per j2.
// NEED: also the least buffer need (Eq. 4) among the rows with those words.
template <bool NEED, class Any>
MMEE_HD void fused_words(const TileTab& tb, const OrderInfo& oi, const DimWords& dw, int c, int capc, Any any, int64_t& words, int& need) {
    const uint32_t f = oi.flags;
    const bool rc = oi.recompute[c] != 0;
    const int64_t rho = rc ? (int64_t)tb.b[LOOP_J] : 1;
    const bool mid_a = rc && (f & (kLaboveI | kJaboveI)) == kJaboveI, mid_b = rc && (f & (kIaboveL | kJaboveL)) == kJaboveL;
    const int A0 = tb.size[S_ik], A1 = tb.size[(f & kLaboveI) ? S_IK : S_iK], B0 = tb.size[S_kl], B1 = tb.size[(f & kIaboveL) ? S_KL : S_Kl];
    const int64_t a0 = dw.ik * tb.b[LOOP_L] * rho, a1 = mid_a ? dw.ik * rho : dw.ik;
    const int64_t b0 = dw.kl * tb.b[LOOP_I] * rho, b1 = mid_b ? dw.kl * rho : dw.kl;
    const int C = tb.size[oi.size_c[c]], D = tb.size[S_lj], E = tb.size[S_ij], Dr = tb.size[oi.size_d_res], Er = tb.size[oi.size_e_res];
    // D and E: both at L3, one held (the better and the other one), both held
    const int64_t d_l3 = dw.lj * tb.b[LOOP_I], e_l3 = dw.ij * tb.b[LOOP_L];
    const int64_t y_held = dw.lj + dw.ij, y_none = d_l3 + e_l3, y_d = dw.lj + e_l3, y_e = d_l3 + dw.ij;
    const bool d_first = y_d <= y_e;
    const int64_t y_best = d_first ? y_d : y_e, y_next = d_first ? y_e : y_d;
    int64_t best = kNoRow;
    int best_need = kSizeCap;
    // A and B with `held` words of room while Op1 runs, `later` of them while Op2 runs, too, fetched with g words
    auto choice = [&](int held, int later, int64_t g) {
        const int s1 = capc - sat_add(held, C), s2 = capc - sat_add(later, C);      // (s1 <= s2)
        const bool f_none = s1 >= 0 && D + E <= s2, f_both = Dr + Er <= s1;
        const bool f_d = Dr <= s1 && Dr + E <= s2, f_e = Er <= s1 && D + Er <= s2;
        if (NEED) {
            // (unsigned: the sums of a choice that does not fit may exceed 2^31)
            auto offer = [&](bool ok, int64_t y, uint32_t d, uint32_t e, uint32_t de) {
                const uint32_t n1 = (uint32_t)held + (uint32_t)C + de, n2 = (uint32_t)C + d + e + (uint32_t)later;
                const int n = (int)(n1 > n2 ? n1 : n2);
                const int64_t w = g + y;
                if (ok && (w < best || (w == best && n < best_need))) { best = w; best_need = n; }
            };
            const uint32_t dr = (uint32_t)Dr, er = (uint32_t)Er;
            offer(f_none, y_none, (uint32_t)D, (uint32_t)E, 0u);
            offer(f_d, y_d, dr, (uint32_t)E, dr);
            offer(f_e, y_e, (uint32_t)D, er, er);
            offer(f_both, y_held, dr, er, dr + er);
        } else {
            int64_t y = f_none ? y_none : kNoRow;
            y = (d_first ? f_e : f_d) ? y_next : y;
            y = (d_first ? f_d : f_e) ? y_best : y;
            y = f_both ? y_held : y;
            best = min64(best, g + y);
        }
    };
    choice(sat_add(A0, B0), 0, a0 + b0);
    choice(sat_add(A1, B0), A1, a1 + b0);
    choice(sat_add(A0, B1), B1, a0 + b1);
    choice(sat_add(A1, B1), sat_add(A1, B1), a1 + b1);
    if (any(mid_a || mid_b)) {
        const int M = !(mid_a || mid_b) ? kSizeCap : tb.size[mid_a ? S_IK : S_KL];
        const int64_t m = mid_a ? dw.ik : dw.kl;
        choice(sat_add(M, mid_a ? B0 : A0), M, m + (mid_a ? b0 : a0));
        choice(sat_add(M, mid_a ? B1 : A1), sat_add(M, mid_a ? B1 : A1), m + (mid_a ? b1 : a1));
    }
    words = best < kNoRow ? best : kNoRow;
    need = best_need;
}

// The same of both nests of an unfused block (any mode), C's write-back in the first and its read-back in the second included.
template <bool NEED>
MMEE_HD void unfused_words(const TileTab& tb, const OrderInfo& oi, const DimWords& dw, int capc, int64_t& words1, int64_t& words2, int& need) {
    const uint32_t f = oi.flags;
    const int s = capc - tb.size[S_il];
    auto least = [&](int p0, int p1, int64_t x0, int64_t x1, int q0, int q1, int64_t y0, int64_t y1, int64_t& words, int& size) {
        words = kNoRow;
        size = kSizeCap;
        auto choice = [&](int room, int64_t w) {        // (sums of two saturated sizes stay below 2^31)
            if (room <= s && (w < words || (NEED && w == words && room < size))) { words = w; size = room; }
        };
        choice(p0 + q0, x0 + y0);
        choice(p1 + q0, x1 + y0);
        choice(p0 + q1, x0 + y1);
        choice(p1 + q1, x1 + y1);
    };
    int64_t x1, x2;
    int u1, u2;
    least(tb.size[S_ik], tb.size[(f & kLaboveI) ? S_IK : S_iK], dw.ik * tb.b[LOOP_L], dw.ik,
          tb.size[S_kl], tb.size[(f & kIaboveL) ? S_KL : S_Kl], dw.kl * tb.b[LOOP_I], dw.kl, x1, u1);
    least(tb.size[S_lj], tb.size[oi.size_d_res], dw.lj * ((f & kIaboveD1) ? tb.b[LOOP_I] : 1u), dw.lj,
          tb.size[S_ij], tb.size[oi.size_e_res], dw.ij * ((f & kLaboveE1) ? tb.b[LOOP_L] : 1u), dw.ij, x2, u2);
    need = tb.size[S_il] + (u1 > u2 ? u1 : u2);
    const bool some = x1 < kNoRow && x2 < kNoRow;
    words1 = some ? x1 + dw.il : kNoRow;
    words2 = some ? x2 + dw.il * ((f & kJaboveC) ? tb.b[LOOP_J] : 1u) : kNoRow;
}

MMEE_HD int64_t edp_bits(int64_t e, int64_t l) {       // ordered by the bit pattern of the positive product
#ifdef __CUDA_ARCH__
    return __double_as_longlong(__dmul_rn((double)e, (double)l));
#else
    const double v = (double)e * (double)l;
    int64_t r;
    __builtin_memcpy(&r, &v, 8);
    return r;
#endif
}

// The objective's key of energy e and latency l; a mapping that violates the cap of a capped objective: kInfKey.
template <int OBJ>
MMEE_HD int64_t key_of(int64_t e, int64_t l, int64_t cap) {
    if (OBJ == MMEE_OBJ_ENERGY) return e;
    if (OBJ == MMEE_OBJ_LATENCY) return l;
    if (OBJ == MMEE_OBJ_EDP) return edp_bits(e, l);
    if (OBJ == MMEE_OBJ_ENERGY_LCAP) return l <= cap ? e : kInfKey;
    return e <= cap ? l : kInfKey;
}

// Key of one mapping of a fused block: x DRAM words, stationary modes of the operators, recomputation factor rho.
template <int OBJ>
MMEE_HD int64_t fused_key(int64_t x, int64_t rho, int64_t P1, int64_t P2, int64_t Q1, int64_t Q2, int64_t c_dram, int64_t cap) {
    return key_of<OBJ>(c_dram * x + P1 * rho + P2, max64(x, Q1 * rho + Q2), cap);
}
// ... of an unfused block: x1, x2 DRAM words of the nests, pass words of the separate softmax pass.
template <int OBJ>
MMEE_HD int64_t unfused_key(int64_t x1, int64_t x2, int64_t pass, int64_t P1, int64_t P2, int64_t Q1, int64_t Q2,
                            int64_t c_dram, int64_t cap) {
    return key_of<OBJ>(c_dram * (x1 + x2 + pass) + P1 + P2, max64(x1, Q1) + pass + max64(x2, Q2), cap);
}

// Least key over the offered stationary pairs (sm_mask bit 3 * sm1 + sm2).  With all nine offered the energy and the
// latency separate into the operators' own minima.
template <int OBJ>
MMEE_HD int64_t fused_least_key(const StatTerms& st, int64_t x, int64_t rho, uint32_t sm_mask, int64_t c_dram, int64_t cap) {
    if ((OBJ == MMEE_OBJ_ENERGY || OBJ == MMEE_OBJ_LATENCY) && sm_mask == 0x1ffu) {
        const int64_t* u = OBJ == MMEE_OBJ_ENERGY ? st.P1 : st.Q1;
        const int64_t* v = OBJ == MMEE_OBJ_ENERGY ? st.P2 : st.Q2;
        const int64_t w = min64(u[0], min64(u[1], u[2])) * rho + min64(v[0], min64(v[1], v[2]));
        return OBJ == MMEE_OBJ_ENERGY ? c_dram * x + w : max64(x, w);
    }
    int64_t best = kInfKey;
#pragma unroll
    for (int s = 0; s < 9; ++s) {
        const int64_t k = fused_key<OBJ>(x, rho, st.P1[s / 3], st.P2[s % 3], st.Q1[s / 3], st.Q2[s % 3], c_dram, cap);
        best = ((sm_mask >> s) & 1u) ? min64(best, k) : best;
    }
    return best;
}
template <int OBJ>
MMEE_HD int64_t unfused_least_key(const StatTerms& st, int64_t x1, int64_t x2, int64_t pass, uint32_t sm_mask, int64_t c_dram,
                                  int64_t cap) {
    if (OBJ == MMEE_OBJ_ENERGY && sm_mask == 0x1ffu)
        return c_dram * (x1 + x2 + pass) + min64(st.P1[0], min64(st.P1[1], st.P1[2])) + min64(st.P2[0], min64(st.P2[1], st.P2[2]));
    if (OBJ == MMEE_OBJ_LATENCY && sm_mask == 0x1ffu)
        return max64(x1, min64(st.Q1[0], min64(st.Q1[1], st.Q1[2]))) + pass + max64(x2, min64(st.Q2[0], min64(st.Q2[1], st.Q2[2])));
    int64_t best = kInfKey;
#pragma unroll
    for (int s = 0; s < 9; ++s) {
        const int64_t k = unfused_key<OBJ>(x1, x2, pass, st.P1[s / 3], st.P2[s % 3], st.Q1[s / 3], st.Q2[s % 3], c_dram, cap);
        best = ((sm_mask >> s) & 1u) ? min64(best, k) : best;
    }
    return best;
}

// No mapping of a tiling has a smaller key: every operand fetched once, C not regenerated, each operator's cheapest and fastest
// stationary mode (of an unfused block: not less DRAM words, not less compute words).
template <int OBJ>
MMEE_HD int64_t tile_least_key(const StatTerms& st, const DimWords& dw, int64_t c_dram, int64_t cap) {
    const int64_t x = dw.ik + dw.kl + dw.lj + dw.ij;
    const int64_t P = min64(st.P1[0], min64(st.P1[1], st.P1[2])) + min64(st.P2[0], min64(st.P2[1], st.P2[2]));
    const int64_t Q = min64(st.Q1[0], min64(st.Q1[1], st.Q1[2])) + min64(st.Q2[0], min64(st.Q2[1], st.Q2[2]));
    return key_of<OBJ>(c_dram * x + P, max64(x, Q), cap);
}

}  // namespace mmee

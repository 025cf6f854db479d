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
};

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

// Rows of a fused block with C at class c: how many fit, and the least DRAM words of one that fits (kNoRow: none).
// With PRUNE only the kept rows are counted (kept[3 * a + b]: bit 4 * d + e); the minimum runs over all rows, which
// changes nothing: a dropped row's keys are never below those of a kept one.
// ANY(x): true if x holds for some lane of the warp (device), for this call (host); a choice of A and B that leaves no
// lane any room is skipped.
// NEED: also the least buffer need (Eq. 4) of a row that fits with the least DRAM words.
template <bool PRUNE, bool NEED, class Any>
MMEE_HD void fused_class(const TileTab& tb, const OrderInfo& oi, const DimWords& dw, int c, int capc,
                         const uint16_t* kept, Any any, uint32_t& rows, int64_t& words, int& need) {
    const int C = tb.size[oi.size_c[c]];
    const int A[3] = {tb.size[S_ik], tb.size[S_iK], tb.size[S_IK]};
    const int B[3] = {tb.size[S_kl], tb.size[S_Kl], tb.size[S_KL]};
    const int D[3] = {tb.size[S_lj], tb.size[oi.size_d_lo], tb.size[S_LJ]};      // L3 and class 1, class 2, class 3
    const int E[3] = {tb.size[S_ij], tb.size[oi.size_e_lo], tb.size[S_IJ]};
    const int Dr = tb.size[oi.size_d_res], Er = tb.size[oi.size_e_res];
    const uint32_t f = oi.flags;
    const bool rc = oi.recompute[c] != 0;
    // DRAM words (Section V-C).  A: fetched again for every l2 (and, when C is regenerated, every j2) above its blocker.
    const int64_t rho = rc ? (int64_t)tb.b[LOOP_J] : 1;
    const int64_t gA[3] = {dw.ik * tb.b[LOOP_L] * rho,
                           dw.ik * ((f & kLaboveI) ? tb.b[LOOP_L] : 1u) * ((f & kJaboveI) ? rho : 1), dw.ik};
    const int64_t gB[3] = {dw.kl * tb.b[LOOP_I] * rho,
                           dw.kl * ((f & kIaboveL) ? tb.b[LOOP_I] : 1u) * ((f & kJaboveL) ? rho : 1), dw.kl};
    // D and E: (both at L3), (one held, the other at L3: the larger and the smaller sum), (both held)
    const int64_t d_l3 = dw.lj * tb.b[LOOP_I], e_l3 = dw.ij * tb.b[LOOP_L];
    const int64_t y_held = dw.lj + dw.ij, y_none = d_l3 + e_l3, y_d = dw.lj + e_l3, y_e = d_l3 + dw.ij;
    const bool d_first = y_d <= y_e;            // holding D saves more
    const int64_t y_best = d_first ? y_d : y_e, y_next = d_first ? y_e : y_d;
    int V[3][3];
#pragma unroll
    for (int x = 0; x < 3; ++x)
#pragma unroll
        for (int y = 0; y < 3; ++y) V[x][y] = D[x] + E[y];          // at most 2^31 - 2
    uint32_t total = 0;
    int64_t best = kNoRow;
    int best_need = kSizeCap;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            // Room for D and E beside A, B, C in each operator's buffer need; A and B count while Op2 runs only from L4
            // on, so that s1 <= s2.  (Sums of two saturated sizes stay below 2^31 and saturate above any capacity.)
            const int s1 = capc - sat_add(sat_add(A[a], B[b]), C);
            const int s2 = capc - sat_add(sat_add(a ? A[a] : 0, b ? B[b] : 0), C);
            if (!any(s1 >= 0 && V[0][0] <= s2)) continue;
            if (PRUNE) {
                uint32_t fit = (s1 >= 0 && V[0][0] <= s2) ? 1u : 0u;
#pragma unroll
                for (int x = 0; x < 3; ++x) {
                    fit |= (D[x] <= s1 && V[x][0] <= s2) ? 1u << (4 * x + 4) : 0u;
                    fit |= (E[x] <= s1 && V[0][x] <= s2) ? 1u << (x + 1) : 0u;
#pragma unroll
                    for (int y = 0; y < 3; ++y) fit |= V[x][y] <= s1 ? 1u << (4 * x + y + 5) : 0u;
                }
                fit &= kept[3 * a + b];
#ifdef __CUDA_ARCH__
                total += (uint32_t)__popc(fit);
#else
                for (; fit; fit &= fit - 1) ++total;
#endif
            } else {
                uint32_t n = 0;
                if (a && b) {
                    // s1 = s2: L3 and the first retained class of D (E) fit together
#pragma unroll
                    for (int x = 0; x < 3; ++x) {
                        uint32_t r = 0;
#pragma unroll
                        for (int y = 0; y < 3; ++y) r += V[x][y] <= s1 ? oi.width[OP_E][y + 1] + (y ? 0u : 1u) : 0u;
                        n += r * (oi.width[OP_D][x + 1] + (x ? 0u : 1u));
                    }
                } else {
                    n = (s1 >= 0 && V[0][0] <= s2) ? 1u : 0u;
#pragma unroll
                    for (int x = 0; x < 3; ++x) {
                        uint32_t r = (D[x] <= s1 && V[x][0] <= s2) ? 1u : 0u;
#pragma unroll
                        for (int y = 0; y < 3; ++y) r += V[x][y] <= s1 ? (uint32_t)oi.width[OP_E][y + 1] : 0u;
                        n += r * oi.width[OP_D][x + 1];
                        n += (E[x] <= s1 && V[0][x] <= s2) ? (uint32_t)oi.width[OP_E][x + 1] : 0u;
                    }
                }
                total += n * (uint32_t)(oi.width[OP_A][a] * oi.width[OP_B][b]);
            }
            const bool f_d = Dr <= s1 && Dr + E[0] <= s2, f_e = Er <= s1 && D[0] + Er <= s2;
            if (NEED) {
                // every choice of D and E by (words, need): where a loop bound is 1 several fetch the same words
                // (unsigned: the sums of a choice that does not fit may exceed 2^31)
                auto offer = [&](bool ok, int64_t y, uint32_t d, uint32_t e, uint32_t held) {
                    const uint32_t n1 = (uint32_t)A[a] + (uint32_t)B[b] + (uint32_t)C + held;
                    const uint32_t n2 = (uint32_t)C + d + e + (a ? (uint32_t)A[a] : 0u) + (b ? (uint32_t)B[b] : 0u);
                    const int n = (int)(n1 > n2 ? n1 : n2);
                    const int64_t w = gA[a] + gB[b] + y;
                    if (ok && (w < best || (w == best && n < best_need))) { best = w; best_need = n; }
                };
                const uint32_t dr = (uint32_t)Dr, er = (uint32_t)Er;
                offer(s1 >= 0 && V[0][0] <= s2, y_none, (uint32_t)D[0], (uint32_t)E[0], 0u);
                offer(f_d, y_d, dr, (uint32_t)E[0], dr);
                offer(f_e, y_e, (uint32_t)D[0], er, er);
                offer(Dr + Er <= s1, y_held, dr, er, dr + er);
                continue;
            }
            int64_t y = (s1 >= 0 && V[0][0] <= s2) ? y_none : kNoRow;
            y = (d_first ? f_e : f_d) ? y_next : y;
            y = (d_first ? f_d : f_e) ? y_best : y;
            y = (Dr + Er <= s1) ? y_held : y;
            best = min64(best, gA[a] + gB[b] + y);
        }
    }
    rows = total * (PRUNE ? 1u : (uint32_t)oi.width[OP_C][c]);
    words = best < kNoRow ? best : kNoRow;
    need = best_need;
}

// Both nests of an unfused block (any mode): feasible rows (of 625, or kept ones) and the least DRAM words of each nest,
// C's write-back in the first and its read-back in the second included.  NEED: as above.
template <bool PRUNE, bool NEED>
MMEE_HD void unfused_nests(const TileTab& tb, const OrderInfo& oi, const DimWords& dw, int capc,
                           uint32_t& fit1, uint32_t& fit2, uint32_t& rows, int64_t& words1, int64_t& words2, int& need) {
    const uint32_t f = oi.flags;
    const int s = capc - tb.size[S_il];
    const int A[3] = {tb.size[S_ik], tb.size[S_iK], tb.size[S_IK]};
    const int B[3] = {tb.size[S_kl], tb.size[S_Kl], tb.size[S_KL]};
    const int D[3] = {tb.size[S_lj], tb.size[oi.size_d_lo], tb.size[S_LJ]};
    const int E[3] = {tb.size[S_ij], tb.size[oi.size_e_lo], tb.size[S_IJ]};
    const int64_t gA[3] = {dw.ik * tb.b[LOOP_L], dw.ik * ((f & kLaboveI) ? tb.b[LOOP_L] : 1u), dw.ik};
    const int64_t gB[3] = {dw.kl * tb.b[LOOP_I], dw.kl * ((f & kIaboveL) ? tb.b[LOOP_I] : 1u), dw.kl};
    const int64_t gD[3] = {dw.lj * ((f & kIaboveD1) ? tb.b[LOOP_I] : 1u), dw.lj * ((f & kIaboveD2) ? tb.b[LOOP_I] : 1u), dw.lj};
    const int64_t gE[3] = {dw.ij * ((f & kLaboveE1) ? tb.b[LOOP_L] : 1u), dw.ij * ((f & kLaboveE2) ? tb.b[LOOP_L] : 1u), dw.ij};
    uint32_t n1 = 0, n2 = 0, m1 = 0, m2 = 0;
    int64_t x1 = kNoRow, x2 = kNoRow;
    int u1 = kSizeCap, u2 = kSizeCap;       // least sizes of the two operands at those words
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const bool o1 = A[a] + B[b] <= s, o2 = D[a] + E[b] <= s;
            if (PRUNE) {
                m1 |= o1 ? 1u << (3 * a + b) : 0u;
                m2 |= o2 ? 1u << (3 * a + b) : 0u;
            } else {
                n1 += o1 ? (uint32_t)(oi.width[OP_A][a] * oi.width[OP_B][b]) : 0u;
                n2 += o2 ? (oi.width[OP_D][a + 1] + (a ? 0u : 1u)) * (oi.width[OP_E][b + 1] + (b ? 0u : 1u)) : 0u;
            }
            if (NEED) {
                const int64_t w1 = gA[a] + gB[b], w2 = gD[a] + gE[b];
                if (o1 && (w1 < x1 || (w1 == x1 && A[a] + B[b] < u1))) { x1 = w1; u1 = A[a] + B[b]; }
                if (o2 && (w2 < x2 || (w2 == x2 && D[a] + E[b] < u2))) { x2 = w2; u2 = D[a] + E[b]; }
            } else {
                x1 = o1 ? min64(x1, gA[a] + gB[b]) : x1;
                x2 = o2 ? min64(x2, gD[a] + gE[b]) : x2;
            }
        }
    fit1 = m1;
    fit2 = m2;
    rows = n1 * n2;
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

}  // namespace mmee

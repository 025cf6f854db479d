// How many rows of a block fit and their least DRAM words, block by block and class by class: what the search's counts of whole
// tilings (count_rows) and its least words (fused_words, unfused_words) are checked against, and what is itself checked against the
// oracle's rows (test_host_math.py).
#pragma once

#include "../paper_2604_03446_b200/csrc/mmee_classes.cuh"

namespace mmee {

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

}  // namespace mmee

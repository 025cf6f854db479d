// The kernels' host/device arithmetic as plain functions, for checks on the CPU (tests/test_host_math.py).
#include "class_forms.h"
#include "../paper_2604_03446_b200/csrc/mmee_eval.cuh"

// Words and cycles of one tile of operator `op` under stationary mode `sm`, and its register-file block.
extern "C" int host_tile_terms(const mmee_workload_t* w, const mmee_arch_t* a, const mmee_objective_t* o, const uint32_t* b,
                               int op, int sm, int64_t out[2], uint32_t blk[3]) {
    mmee::Plan p;
    const int rc = mmee::build_plan(w, a, o, &p);
    if (rc) return rc;
    mmee::tile_array_terms(p, mmee::PlanDivisors{p}, b, op, sm, out[0], out[1], blk);
    return MMEE_OK;
}

// What the search's closed forms over classes of levels give for tiling `t`, order slot `slot`: out[c] = {first level of C's
// class, levels in it, rows that fit, least words, need of the words; rows and words as counted without the need; rows that
// pruning keeps} for the three classes of C, then out[3] = the same of an unfused block ({0, 5, rows, words of the first nest,
// need, rows, words of the second nest, kept rows of mode 1}).
extern "C" int host_classes(const mmee_workload_t* w, const mmee_arch_t* a, const mmee_objective_t* o, uint32_t t, int slot,
                            int64_t out[4][8]) {
    using namespace mmee;
    Plan p;
    uint32_t kept;
    int rc = build_plan(w, a, o, &p);
    KeptMasks masks;
    if (rc || (rc = find_kept_masks(p, &masks, &kept))) return rc;
    TileTab tb = {};
    for (int d = 3; d >= 0; --d) {
        const uint32_t g = p.divs[d][t % p.ndiv[d]];
        t /= p.ndiv[d];
        tb.b[4 + d] = g;
        tb.b[d] = p.dim[d] / g;
    }
    for (int i = 0; i < kSizeSlots; ++i) tb.size[i] = sat_size(size_words(p.dim, tb.b + 4, i));
    const int64_t I = p.dim[0], K = p.dim[1], L = p.dim[2], J = p.dim[3];
    const DimWords dw = {I * K, K * L, L * J, I * J, I * L};
    const OrderInfo& oi = p.order[slot];
    const int cap = (int)p.cap_words;
    auto any = [](bool v) { return v; };
    int need, unused;
    uint32_t rows, fit1, fit2;
    for (int c = 0; c < 3; ++c) {
        out[c][0] = oi.first[OP_C][c];
        out[c][1] = oi.width[OP_C][c];
        fused_class<false, true>(tb, oi, dw, c, cap, nullptr, any, rows, out[c][3], need);
        out[c][2] = rows;
        out[c][4] = need;
        fused_class<false, false>(tb, oi, dw, c, cap, nullptr, any, rows, out[c][6], unused);
        out[c][5] = rows;
        int64_t x;
        fused_class<true, false>(tb, oi, dw, c, cap, masks.fused[slot][c], any, rows, x, unused);
        out[c][7] = rows;
        if (x != out[c][6]) return MMEE_ERR_CHECK;
    }
    out[3][0] = 0;
    out[3][1] = 5;
    unfused_nests<false, true>(tb, oi, dw, cap, fit1, fit2, rows, out[3][3], out[3][6], need);
    out[3][2] = rows;
    out[3][4] = need;
    int64_t x1, x2;
    unfused_nests<false, false>(tb, oi, dw, cap, fit1, fit2, rows, x1, x2, unused);
    out[3][5] = rows;
    if (x1 != out[3][3] || x2 != out[3][6]) return MMEE_ERR_CHECK;
    unfused_nests<true, false>(tb, oi, dw, cap, fit1, fit2, rows, x1, x2, unused);
    out[3][7] = 0;
    for (int ab = 0; ab < 9; ++ab)
        if ((fit1 >> ab) & 1u) out[3][7] += __builtin_popcount(fit2 & masks.unfused[0][slot][ab]);
    return x1 == out[3][3] && x2 == out[3][6] ? MMEE_OK : MMEE_ERR_CHECK;
}

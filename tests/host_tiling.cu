// The search's counts and least words of whole tilings beside the same by blocks and classes, for a check on the CPU
// (tests/test_host_tiling.py).
#include "class_forms.h"

namespace {

using namespace mmee;

// Whether a tiling's bound is not above the least key of one of its items, whatever the accelerator: stationary-pair terms, energy of
// a DRAM word, bound on the other key and offered pairs drawn from `seed`.  (x1 + x2: an unfused block.)
template <int OBJ>
bool bound_holds(const DimWords& dw, int64_t x1, int64_t x2, bool fused, int64_t rho, uint64_t seed) {
    auto next = [&](uint64_t n) {
        seed = seed * 6364136223846793005ull + 1442695040888963407ull;
        return (int64_t)((seed >> 33) % n);
    };
    const int64_t scale = (int64_t)1 << next(24);
    StatTerms st;
    for (int i = 0; i < 3; ++i) { st.P1[i] = next(scale); st.P2[i] = next(scale); st.Q1[i] = next(scale); st.Q2[i] = next(scale); }
    const int64_t c_dram = next(4) ? next(300) : 0, pass = fused || next(2) ? 0 : 2 * dw.il;
    const uint32_t mask = next(2) ? 0x1ffu : (uint32_t)(1 + next(511));
    // a bound near what the item has of the other key, so that it decides
    const int64_t other = OBJ == MMEE_OBJ_ENERGY_LCAP ? x1 + x2 + st.Q1[0] : c_dram * (x1 + x2) + st.P1[0];
    const int64_t cap = next(3) ? other * next(200) / 100 : INT64_MAX - 1;
    const int64_t least = tile_least_key<OBJ>(st, dw, c_dram, cap);
    const int64_t key = fused ? fused_least_key<OBJ>(st, x1, rho, mask, c_dram, cap)
                              : unfused_least_key<OBJ>(st, x1, x2, pass, mask, c_dram, cap);
    return least <= key;
}
bool bounds_hold(const DimWords& dw, int64_t x1, int64_t x2, bool fused, int64_t rho, uint64_t seed) {
    return bound_holds<MMEE_OBJ_ENERGY>(dw, x1, x2, fused, rho, seed) && bound_holds<MMEE_OBJ_LATENCY>(dw, x1, x2, fused, rho, seed + 1) &&
           bound_holds<MMEE_OBJ_EDP>(dw, x1, x2, fused, rho, seed + 2) && bound_holds<MMEE_OBJ_ENERGY_LCAP>(dw, x1, x2, fused, rho, seed + 3) &&
           bound_holds<MMEE_OBJ_LATENCY_ECAP>(dw, x1, x2, fused, rho, seed + 4);
}

}  // namespace

// Every `stride`-th tiling of a problem: the rows of all its blocks that fit, all of them and the kept ones, every block's least words
// and needs, and the tiling's bounds on keys and needs.  Returns MMEE_OK, or MMEE_ERR_CHECK with the tiling in *at where two of them
// differ or a bound is above what it bounds.
extern "C" int host_tilings(const mmee_workload_t* w, const mmee_arch_t* a, const mmee_objective_t* o, uint32_t stride, uint64_t* at) {
    using namespace mmee;
    Plan p;
    uint32_t n_kept;
    int rc = build_plan(w, a, o, &p);
    KeptMasks masks;
    if (rc || (rc = find_kept_masks(p, &masks, &n_kept)) || (rc = set_kept_weights(&p, &n_kept))) return rc;
    const CountWeights all = count_weights((int)p.n_orders);
    CountWeights kept = {};
    for (int i = 0; i < (int)(sizeof(kept) / 4); ++i) (&kept.w[0][0][0])[i] = p.kept_weights[i / 8] >> (4 * (i % 8)) & 15u;
    const int64_t I = p.dim[0], K = p.dim[1], L = p.dim[2], J = p.dim[3];
    const DimWords dw = {I * K, K * L, L * J, I * J, I * L};
    const int cap = (int)p.cap_words;
    const uint32_t modes = (p.fuse_mask >> 1 & 1u) + (p.fuse_mask >> 2 & 1u);
    auto any = [](bool v) { return v; };
    for (uint64_t tiling = 0; tiling < p.n_tilings; tiling += stride) {
        *at = tiling;
        TileTab tb = {};
        uint64_t t = tiling;
        for (int d = 3; d >= 0; --d) {
            tb.b[4 + d] = p.divs[d][t % p.ndiv[d]];
            tb.b[d] = p.dim[d] / tb.b[4 + d];
            t /= p.ndiv[d];
        }
        for (int i = 0; i < kSizeSlots; ++i) tb.size[i] = sat_size(size_words(p.dim, tb.b + 4, i));
        uint64_t rows = 0, rows_kept = 0, want = 0, want_kept = 0;
        // (no row needs less buffer: every operand at L3)
        const int one = sat_add(tb.size[S_ik], tb.size[S_kl]), two = sat_add(tb.size[S_lj], tb.size[S_ij]);
        const int least_need = sat_add(tb.size[S_il], one > two ? one : two);
        const int c0 = (p.fuse_mask & 1u) ? 0 : 4, c1 = modes ? 5 : 4;
        for (int ab = 0; ab < 9; ++ab) {
            rows += count_rows(tb.size, ab, c0, c1, modes, cap, all, p.n_orders == 2, any);
            for (int c = c0; c < c1; ++c) rows_kept += count_rows(tb.size, ab, c, c + 1, 1u, cap, kept, p.n_orders == 2, any);
        }
        for (uint32_t s = 0; s < p.n_orders; ++s) {
            uint32_t n, fit1, fit2;
            int64_t x, x2, y, y2;
            int need, need2;
            for (int c = 0; c < 3 && (p.fuse_mask & 1u); ++c) {
                fused_class<false, true>(tb, p.order[s], dw, c, cap, nullptr, any, n, x, need);
                want += n;
                fused_words<true>(tb, p.order[s], dw, c, cap, any, y, need2);
                if (x != y || (x < kNoRow && need != need2)) return MMEE_ERR_CHECK;
                if (x < kNoRow && (need < least_need ||
                                   !bounds_hold(dw, x, 0, true, p.order[s].recompute[c] ? tb.b[LOOP_J] : 1, tiling * 97 + s * 3 + c)))
                    return MMEE_ERR_CHECK;
                fused_words<false>(tb, p.order[s], dw, c, cap, any, y, need2);
                if (x != y) return MMEE_ERR_CHECK;
                fused_class<true, false>(tb, p.order[s], dw, c, cap, masks.fused[s][c], any, n, x, need);
                want_kept += n;
            }
            if (!modes) continue;
            unfused_nests<false, true>(tb, p.order[s], dw, cap, fit1, fit2, n, x, x2, need);
            want += (uint64_t)n * modes;
            unfused_words<true>(tb, p.order[s], dw, cap, y, y2, need2);
            if (x != y || x2 != y2 || (x < kNoRow && need != need2)) return MMEE_ERR_CHECK;
            if (x < kNoRow && (need < least_need || !bounds_hold(dw, x, x2, false, 1, tiling * 97 + s * 3 + 50))) return MMEE_ERR_CHECK;
            unfused_words<false>(tb, p.order[s], dw, cap, y, y2, need2);
            if (x != y || x2 != y2) return MMEE_ERR_CHECK;
            unfused_nests<true, false>(tb, p.order[s], dw, cap, fit1, fit2, n, x, x2, need);
            for (uint32_t phi = 1; phi <= 2; ++phi)
                for (int ab = 0; ab < 9 && ((p.fuse_mask >> phi) & 1u); ++ab)
                    if ((fit1 >> ab) & 1u) want_kept += (uint64_t)__builtin_popcount(fit2 & masks.unfused[phi - 1][s][ab]);
        }
        if (rows != want || rows_kept != want_kept) return MMEE_ERR_CHECK;
    }
    return MMEE_OK;
}

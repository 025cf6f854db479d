// Offline symbolic row pruning for single-optimum searches (Section VI-B), in a tie-safe form.
//
// The paper drops a row v when another row u of the same group needs no more buffer and no less
// DRAM traffic for every tiling, one of the two strictly (Eq. 12).  That keeps the optimum VALUE but
// may drop a row that merely ties with a kept one, and this library promises the lowest index among
// equal keys.  The rule used here is therefore: v is dropped iff some row u of the same fusion mode
// and recompute group with a LOWER row index has, symbolically, BS^Op1_u <= BS^Op1_v,
// BS^Op2_u <= BS^Op2_v and DA_u <= DA_v (for unfused rows: the DRAM sums of the two operators
// separately).  Then for every tiling and stationary pair u fits whenever v fits and
// (key_u, idx_u) < (key_v, idx_v) under each objective (energy is a sum, latency a max / a sum of
// maxima, EDP their product: all monotone), so v can never be the optimum.  Rows with identical
// symbolic sums are dropped too, except the one with the lowest index.  Valid for k = 1 only.
#include "mmee_plan.h"

#include <algorithm>
#include <cstring>
#include <map>
#include <mutex>
#include <vector>

namespace mmee {

namespace {

// A sum of monomials; each monomial is the set of loop bounds (query vector) it multiplies.
struct SymSum {
    int n = 0;
    uint8_t term[6] = {0, 0, 0, 0, 0, 0};
    void add(uint8_t q) { term[n++] = q; }
    void canon() { std::sort(term, term + n); }
    bool operator<(const SymSum& o) const {
        if (n != o.n) return n < o.n;
        for (int i = 0; i < n; ++i) if (term[i] != o.term[i]) return term[i] < o.term[i];
        return false;
    }
};

// q <= p for every assignment of bounds >= 1 if q's terms embed one-to-one into supersets among p's.
bool embeds(const SymSum& p, const SymSum& q, int qi, unsigned used) {
    if (qi == q.n) return true;
    for (int i = 0; i < p.n; ++i) {
        if (used & (1u << i)) continue;
        if ((q.term[qi] & p.term[i]) != q.term[qi]) continue;
        if (embeds(p, q, qi + 1, used | (1u << i))) return true;
    }
    return false;
}
bool sum_le(const SymSum& q, const SymSum& p) { return q.n <= p.n && embeds(p, q, 0, 0); }

struct Signature {
    SymSum part[4];       // BS^Op1, BS^Op2, DA (fused) or DA of Op1, DA of Op2 (unfused; part[3] empty when fused)
    int group;            // fusion mode * 2 + recompute flag
    bool operator<(const Signature& o) const {
        if (group != o.group) return group < o.group;
        for (int i = 0; i < 4; ++i) {
            if (part[i] < o.part[i]) return true;
            if (o.part[i] < part[i]) return false;
        }
        return false;
    }
};

bool sig_le(const Signature& u, const Signature& v) {
    if (u.group != v.group) return false;
    for (int i = 0; i < 4; ++i) if (!sum_le(u.part[i], v.part[i])) return false;
    return true;
}

Signature signature_of(const QueryTables& q, uint32_t phi, uint32_t order, const uint32_t lv[5]) {
    Signature s;
    const bool fused = phi == 0;
    const uint32_t rc = fused ? q.recompute[order][lv[OP_C]] : 0u;
    s.group = (int)(phi * 2 + rc);
    uint8_t bs[5];
    for (int x = 0; x < 5; ++x) bs[x] = q.bs[order][x][lv[x]];
    s.part[0].add(bs[OP_A]); s.part[0].add(bs[OP_B]); s.part[0].add(bs[OP_C]);
    s.part[1].add(bs[OP_C]); s.part[1].add(bs[OP_D]); s.part[1].add(bs[OP_E]);
    if (fused) {
        if (lv[OP_D]) s.part[0].add(bs[OP_D]);
        if (lv[OP_E]) s.part[0].add(bs[OP_E]);
        if (lv[OP_A]) s.part[1].add(bs[OP_A]);
        if (lv[OP_B]) s.part[1].add(bs[OP_B]);
        s.part[2].add(q.da[order][OP_A][lv[OP_A]][rc]);
        s.part[2].add(q.da[order][OP_B][lv[OP_B]][rc]);
        s.part[2].add(q.da[order][OP_D][lv[OP_D]][0]);
        s.part[2].add(q.da[order][OP_E][lv[OP_E]][0]);
    } else {
        s.part[2].add(q.da_unfused[order][OP_A][lv[OP_A]]);
        s.part[2].add(q.da_unfused[order][OP_B][lv[OP_B]]);
        s.part[3].add(q.da_unfused[order][OP_C][0]);
        s.part[3].add(q.da_unfused[order][OP_D][lv[OP_D]]);
        s.part[3].add(q.da_unfused[order][OP_E][lv[OP_E]]);
    }
    for (int i = 0; i < 4; ++i) s.part[i].canon();
    return s;
}

}  // namespace

namespace {

// Fills keep[row] (rows_per_tiling entries) for the plan's row space.
void build_row_keep(const Plan& p, std::vector<uint8_t>* keep) {
    const uint32_t R = p.rows_per_tiling;
    keep->assign(R, 1);
    std::vector<int> sig_of_row(R);
    std::map<Signature, int> ids;
    std::vector<Signature> sigs;
    std::vector<uint32_t> first_row;                      // lowest row index with this signature
    // rows in index order: fused r = o*3125 + lA*625 + lB*125 + lC*25 + lD*5 + lE, then per unfused
    // mode o*625 + lA*125 + lB*25 + lD*5 + lE
    const uint32_t fused_rows = p.n_fused_blocks * 3125u;
    for (uint32_t row = 0; row < R; ++row) {
        uint32_t block, lv[5];
        if (row < fused_rows) {
            block = row / 3125u;
            const uint32_t r = row % 3125u;
            lv[0] = r / 625u; lv[1] = (r / 125u) % 5u; lv[2] = (r / 25u) % 5u; lv[3] = (r / 5u) % 5u; lv[4] = r % 5u;
        } else {
            const uint32_t u = row - fused_rows;
            block = p.n_fused_blocks + u / 625u;
            const uint32_t r = u % 625u;
            lv[0] = r / 125u; lv[1] = (r / 25u) % 5u; lv[2] = 0; lv[3] = (r / 5u) % 5u; lv[4] = r % 5u;
        }
        const uint32_t phi = p.block_phi[block], order = p.order_id[p.block_order_slot[block]];
        {
            const Signature s = signature_of(p.q, phi, order, lv);
            auto it = ids.find(s);
            if (it == ids.end()) {
                it = ids.emplace(s, (int)sigs.size()).first;
                sigs.push_back(s);
                first_row.push_back(row);
            }
            sig_of_row[row] = it->second;
        }
    }
    // best_row[s] = lowest row index among the signatures that are <= s (itself included)
    const size_t n = sigs.size();
    std::vector<uint32_t> best_row(first_row);
    for (size_t v = 0; v < n; ++v)
        for (size_t u = 0; u < n; ++u)
            if (first_row[u] < best_row[v] && sig_le(sigs[u], sigs[v])) best_row[v] = first_row[u];
    for (uint32_t row = 0; row < R; ++row)
        if (best_row[sig_of_row[row]] < row) (*keep)[row] = 0;
}

}  // namespace

void row_pruning_keep(const Plan& p, uint8_t* out, uint32_t* kept_rows) {
    std::vector<uint8_t> keep;
    build_row_keep(p, &keep);
    *kept_rows = 0;
    for (uint32_t r = 0; r < p.rows_per_tiling; ++r) { out[r] = keep[r]; *kept_rows += keep[r]; }
}

// The kept rows as masks over classes of levels.  A row that is not the first of its class combination has equal
// buffer needs and DRAM words as that first row and a higher index, so it is never kept; MMEE_ERR_CHECK if it were.
int find_kept_masks(const Plan& p, KeptMasks* masks, uint32_t* kept_rows) {
    std::vector<uint8_t> keep(p.rows_per_tiling);
    row_pruning_keep(p, keep.data(), kept_rows);
    *masks = {};
    for (uint32_t row = 0; row < p.rows_per_tiling; ++row) {
        if (!keep[row]) continue;
        const uint32_t task = row / 125u, mid = row % 125u / 25u, de = row % 25u;
        const bool fused = task < p.fused_tasks;
        const uint32_t u = fused ? task : task - p.fused_tasks, per = fused ? 25u : 5u;
        const uint32_t block = fused ? u / per : p.n_fused_blocks + u / per;
        const uint32_t slot = p.block_order_slot[block];
        const OrderInfo& o = p.order[slot];
        const uint32_t lv[5] = {fused ? u % 25u / 5u : u % 5u, fused ? u % 5u : mid, fused ? mid : 0u, de / 5u, de % 5u};
        uint32_t cls[5];
        for (int x = 0; x < 5; ++x) {
            int c = -1;
            for (int i = 0; i < 4; ++i) if (o.width[x][i] && o.first[x][i] == lv[x]) c = i;
            if (c < 0) return MMEE_ERR_CHECK;
            cls[x] = (uint32_t)c;
        }
        if (fused) {
            masks->fused[slot][cls[OP_C]][3 * cls[OP_A] + cls[OP_B]] |= (uint16_t)(1u << (4 * cls[OP_D] + cls[OP_E]));
        } else {
            // an unfused nest knows no retained operands: L3 and the class from L4 on are one class of D and of E
            if (cls[OP_D] == 1 || cls[OP_E] == 1) return MMEE_ERR_CHECK;
            const uint32_t d = cls[OP_D] ? cls[OP_D] - 1 : 0, e = cls[OP_E] ? cls[OP_E] - 1 : 0;
            masks->unfused[p.block_phi[block] - 1][slot][3 * cls[OP_A] + cls[OP_B]] |= (uint16_t)(1u << (3 * d + e));
        }
    }
    return MMEE_OK;
}

// The same as weights of a tiling's count, [3 * a + b][size slot of C, or 4 for an unfused mode][choice of D and E]: at most twelve
// rows (two modes of six orders) have one.
static int find_kept_weights(Plan* p, uint32_t* kept_rows) {
    KeptMasks masks;
    const int rc = find_kept_masks(*p, &masks, kept_rows);
    if (rc) return rc;
    std::memset(p->kept_weights, 0, sizeof(p->kept_weights));
    static_assert(9 * 5 * kCountChoices <= 8 * sizeof(p->kept_weights) / 4, "four bits each");
    for (uint32_t slot = 0; slot < p->n_orders; ++slot) {
        const OrderInfo& o = p->order[slot];
        const int d_lo = o.size_d_lo - S_lj, e_lo = o.size_e_lo - S_ij;
        auto add = [&](int ab, int c, int de) {
            const int at = (ab * 5 + c) * kCountChoices + de;
            p->kept_weights[at / 8] += 1u << (4 * (at % 8));
        };
        for (int ab = 0; ab < 9; ++ab) {
            for (int c = 0; c < 3; ++c)
                for (int de = 0; de < 16; ++de)
                    if (masks.fused[slot][c][ab] >> de & 1) add(ab, o.size_c[c] - S_il, de_choice(de / 4, de % 4, d_lo, e_lo));
            for (int mode = 0; mode < 2; ++mode)
                for (int de = 0; de < 9; ++de)
                    if (masks.unfused[mode][slot][ab] >> de & 1) add(ab, 4, de_choice(de / 3 + 1, de % 3 + 1, d_lo, e_lo));
        }
    }
    return MMEE_OK;
}

// They depend on the orders and the fusion modes alone, not on the problem: like the paper's offline pruning they are
// found once for each of the 14 choices (13 ms of host time) and kept.
int set_kept_weights(Plan* p, uint32_t* kept_rows) {
    struct Entry {
        std::once_flag once;
        int status = MMEE_OK;
        uint32_t rows = 0;
        uint32_t weights[sizeof(Plan::kept_weights) / 4] = {};
    };
    static Entry entries[2][8];
    Entry& e = entries[p->n_orders == kMaxOrders ? 1 : 0][p->fuse_mask & 7u];
    std::call_once(e.once, [&] {
        e.status = find_kept_weights(p, &e.rows);
        std::memcpy(e.weights, p->kept_weights, sizeof(e.weights));
    });
    std::memcpy(p->kept_weights, e.weights, sizeof(e.weights));
    *kept_rows = e.rows;
    return e.status;
}

}  // namespace mmee

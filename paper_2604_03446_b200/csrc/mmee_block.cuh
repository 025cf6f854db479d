// One block of mappings (tiling, fusion mode, order) level by level: the tables from which single rows and mappings are
// evaluated exactly -- the winners' blocks at the end of a search, the key dump, the group flags.  Unlike the search's
// closed forms over classes (mmee_classes.cuh) these terms come from the query vectors, exp(q . ln b) (Eq. 8).
#pragma once

#include "mmee_classes.cuh"
#include "mmee_eval.cuh"

namespace mmee {

struct BlockTab {
    int32_t  size[5][5];        // buffer words by operand and level, saturated to kSizeCap
    uint32_t phi, slot;         // fusion mode, order slot
    uint32_t t, jD;
    int64_t  g[5][5][2];        // DRAM words by operand, level and recompute flag ([2][0]: C read back, unfused)
    int64_t  P1[3], P2[3], Q1[3], Q2[3];      // as in TileTab
    int64_t  c_write, pass;     // unfused: words of C's write-back, of the separate softmax pass
    uint64_t first_idx;         // index of the block's first mapping
};

constexpr int kBlockItems = 32;

// The bounds of a search: the plan's, or one of them set by the search before it (see LaunchShape::chain).
struct Limits { int64_t cap_words, key_cap; };


// Stationary-mode terms of one operator of one tiling: its energy and compute words at rho = 1 (see TileTab).
template <class Divisors>
__device__ __forceinline__ void stationary_terms(const Plan& p, const Divisors& dv, const uint32_t b[8], int op, int sm, int64_t& P, int64_t& Q) {
    int64_t w, cy;
    uint32_t blk[3];
    tile_array_terms(p, dv, b, op, sm, w, cy, blk);
    // tile invocations; partial sums carried between the steps of the reduction; MACs (see tiling_counts)
    const int64_t il = (int64_t)b[LOOP_I] * b[LOOP_L];
    const int64_t outer = op == 0 ? il : (int64_t)b[LOOP_I] * b[LOOP_J];
    const int64_t calls = il * (op == 0 ? b[LOOP_K] : b[LOOP_J]);
    const int64_t carried = (calls - outer) * b[4 + LOOP_I] * (op == 0 ? b[4 + LOOP_L] : b[4 + LOOP_J]);
    const int64_t elements = (int64_t)p.dim[LOOP_I] * p.dim[LOOP_L];
    P = p.c_br * (calls * w + carried) + p.c_mac * (elements * (op == 0 ? p.dim[LOOP_K] : p.dim[LOOP_J])) + (op == 0 ? p.c_sfu * elements : 0);
    Q = calls * cy * (int64_t)p.bw;
}

// Index of the first mapping of block `id` = tiling * n_blocks + block.
__device__ __forceinline__ uint64_t block_first_idx(const Plan& p, uint32_t id) {
    const uint32_t t = id / p.n_blocks, block = id - t * p.n_blocks;
    const uint32_t fused_rows = p.n_fused_blocks * 3125u;
    const uint32_t row0 = block < p.n_fused_blocks ? block * 3125u : fused_rows + (block - p.n_fused_blocks) * 625u;
    return ((uint64_t)t * p.rows_per_tiling + row0) * 9u;
}

// Item `item` (0 .. kBlockItems - 1) of the tables of block `id` = tiling * n_blocks + block.
template <class Divisors>
__device__ __forceinline__ void block_item(const Plan& p, const Divisors& dv, uint32_t id, int item, BlockTab* bt) {
    const uint32_t t = id / p.n_blocks, block = id - t * p.n_blocks;
    const uint32_t phi = p.block_phi[block], slot = p.block_order_slot[block], order = p.order_id[slot];
    uint32_t b[8];
    tiling_bounds(p, dv, t, b);
    if (item < 25) {
        const int x = item / 5, l = item % 5;
        bt->size[x][l] = sat_size((uint64_t)monomial(p.q.bs[order][x][l], b));
        int64_t g0 = 0, g1 = 0;
        if (phi) g0 = g1 = monomial(p.q.da_unfused[order][x][l], b);
        else if (x != OP_C) { g0 = monomial(p.q.da[order][x][l][0], b); g1 = monomial(p.q.da[order][x][l][1], b); }
        bt->g[x][l][0] = g0;
        bt->g[x][l][1] = g1;
    } else if (item < 31) {
        const int op = (item - 25) / 3, sm = (item - 25) % 3;
        int64_t P, Q;
        stationary_terms(p, dv, b, op, sm, P, Q);
        (op ? bt->P2 : bt->P1)[sm] = P;
        (op ? bt->Q2 : bt->Q1)[sm] = Q;
    } else {
        const int64_t il = (int64_t)p.dim[LOOP_I] * p.dim[LOOP_L];
        bt->phi = phi;
        bt->slot = slot;
        bt->t = t;
        bt->jD = b[LOOP_J];
        bt->c_write = il;
        bt->pass = phi == 2 ? 2 * il : 0;
        bt->first_idx = block_first_idx(p, id);
    }
}

// One row of the block: levels (beta - 3) of A, B, C, D, E (C's is 0 when unfused).
struct RowTerms {
    bool fits;
    int64_t need;               // buffer words (Eq. 4)
    int64_t x1, x2;             // DRAM words of A and B, of D and E (unfused: C's write-back and read-back included)
    int64_t rho;                // recomputation factor of C
};
__device__ __forceinline__ RowTerms row_terms(const Plan& p, const Limits& lim, const BlockTab& bt, int a, int b, int c, int d, int e) {
    RowTerms r;
    const int64_t A = bt.size[0][a], B = bt.size[1][b], C = bt.size[2][c], D = bt.size[3][d], E = bt.size[4][e];
    int64_t need1 = A + B + C, need2 = C + D + E;
    int rc = 0;
    if (bt.phi == 0) {
        need1 += (d ? D : 0) + (e ? E : 0);
        need2 += (a ? A : 0) + (b ? B : 0);
        rc = p.q.recompute[p.order_id[bt.slot]][c];
    }
    r.need = max64(need1, need2);
    r.fits = r.need <= lim.cap_words;
    r.rho = rc ? (int64_t)bt.jD : 1;
    r.x1 = bt.g[0][a][rc] + bt.g[1][b][rc];
    r.x2 = bt.g[3][d][0] + bt.g[4][e][0];
    if (bt.phi) { r.x1 += bt.c_write; r.x2 += bt.g[2][0][0]; }
    return r;
}

template <int OBJ>
__device__ __forceinline__ int64_t mapping_key(const Plan& p, const Limits& lim, const BlockTab& bt, const RowTerms& r, int s) {
    const int u = s / 3, v = s - 3 * u;
    return bt.phi == 0 ? fused_key<OBJ>(r.x1 + r.x2, r.rho, bt.P1[u], bt.P2[v], bt.Q1[u], bt.Q2[v], p.c_dram_gb, lim.key_cap)
                       : unfused_key<OBJ>(r.x1, r.x2, bt.pass, bt.P1[u], bt.P2[v], bt.Q1[u], bt.Q2[v], p.c_dram_gb, lim.key_cap);
}

// Row `row` of the block by its levels; the number of rows of the block.
__device__ __forceinline__ RowTerms block_row(const Plan& p, const Limits& lim, const BlockTab& bt, uint32_t row) {
    const int e = (int)(row % 5u), d = (int)(row / 5u % 5u);
    if (bt.phi == 0) return row_terms(p, lim, bt, (int)(row / 625u), (int)(row / 125u % 5u), (int)(row / 25u % 5u), d, e);
    return row_terms(p, lim, bt, (int)(row / 125u), (int)(row / 25u % 5u), 0, d, e);
}
__device__ __forceinline__ uint32_t block_rows(const BlockTab& bt) { return bt.phi == 0 ? 3125u : 625u; }

}  // namespace mmee

// Internal: the search plan handed to the kernels by value, and the host planner's interface.
#pragma once

#include <stdint.h>
#include "../../include/mmee.h"

namespace mmee {

constexpr int kMaxOrders = 6;
constexpr int kMaxBlocks = 18;     // (fusion mode, order) pairs
constexpr int kRowsPerTask = 125;   // one middle level (C when fused, B when unfused) x levels of D and E
constexpr int kCandPerTask = 1125;  // rows x 9 stationary pairs
constexpr int64_t kInfKey = INT64_MAX;

// Model arithmetic that the host can run as well as the kernels.
#ifdef __CUDACC__
#define MMEE_HD __host__ __device__ __forceinline__
#else
#define MMEE_HD inline
#endif

// Operand / loop numbering shared by host planner and kernels.
enum { OP_A = 0, OP_B = 1, OP_C = 2, OP_D = 3, OP_E = 4 };
enum { LOOP_I = 0, LOOP_K = 1, LOOP_L = 2, LOOP_J = 3 };

// Query vectors as 8-bit selector masks over b = [i_D,k_D,l_D,j_D,i_G,k_G,l_G,j_G]
// (bit d = x_D of loop d, bit 4+d = x_G).  Indexed by the ACTUAL order id 0..5.
struct QueryTables {
    uint8_t bs[6][5][5];          // [order][operand][beta-3]            operand buffer size
    uint8_t da[6][5][5][2];       // [order][operand][beta-3][recompute] fused DRAM access (C unused)
    uint8_t da_unfused[6][5][5];  // [order][operand][beta-3]            unfused; C: read-back at beta=3
    uint8_t recompute[6][5];      // [order][beta_C-3]
};

// Buffer sizes of a tiling's operands (TileTab::size): lower case a tile extent, upper case the whole dimension.
enum SizeSlot { S_ik, S_iK, S_IK, S_kl, S_Kl, S_KL, S_il, S_Il, S_iL, S_IL, S_lj, S_Lj, S_lJ, S_LJ, S_ij, S_Ij, S_iJ, S_IJ, kSizeSlots };

// Levels of one operand fall into classes with equal buffer need and equal DRAM words: only the operand's own inter-tile
// loops change either (Section V-B, V-C), plus the step from L3 to L4, from where the operand counts as retained while
// the other operator runs (Eq. 1, 2) and D / E leave Scenario 2.  Classes, in ascending level order:
//   A: L3 | L4 .. below i2 | i2 ..          B: L3 | L4 .. below l2 | l2 ..
//   C: L3 .. below its lower own loop | .. below its upper one | upper ..
//   D, E: L3 | L4 .. below the lower own loop | .. below the upper one | upper ..
struct alignas(4) OrderInfo {
    uint8_t first[5][4];          // first level (beta - 3) of each class; classes per operand: 3, 3, 3, 4, 4
    uint8_t width[5][4];          // levels in the class (0 for a fourth class that does not exist)
    uint8_t recompute[3];         // C is regenerated, by class of C
    uint8_t size_c[3];            // where a class's buffer size sits in a tiling's size table (TileTab::size): C by
    uint8_t size_d_lo, size_e_lo; // class; D / E with the lower own loop resident (class 2)
    uint8_t size_d_res, size_e_res;   // the smallest class of D / E that is fetched only once
    uint16_t flags;               // OrderFlag bits: which loops run above which
};
enum OrderFlag {
    kLaboveI = 1, kJaboveI = 2, kIaboveL = 4, kJaboveL = 8,
    kJaboveC = 16,                // j2 above the lower own loop of C
    kIaboveD1 = 32, kIaboveD2 = 64,   // i2 above the lower / upper own loop of D
    kLaboveE1 = 128, kLaboveE2 = 256  // l2 above the lower / upper own loop of E
};
// Rows kept by symbolic pruning, by classes (every kept row is the first of its class combination).
struct KeptMasks {
    uint16_t fused[kMaxOrders][3][9];         // [order slot][class of C][3 * class of A + class of B]: bit 4 * d + e
    uint16_t unfused[2][kMaxOrders][9];       // [unfused mode][order slot][3 * a + b]: bit 3 * d + e (L3, L4 merged)
};

// Where a tiling's count keeps rows with D and E of classes d, e (0: L3, 1..3), by their size slots (CountWeights): 4 * x + y both
// retained, 16 + x D retained and E at L3, 20 + y the other way round, 24 both at L3.  `lo`: the size slot of class 2 behind that
// of class 1, 1 or 2.
MMEE_HD constexpr int de_choice(int d, int e, int d_lo, int e_lo) {
    return d && e ? 4 * (d == 3 ? 3 : (d == 2 ? d_lo : 0)) + (e == 3 ? 3 : (e == 2 ? e_lo : 0))
                  : (d ? 16 + (d == 3 ? 3 : (d == 2 ? d_lo : 0)) : (e ? 20 + (e == 3 ? 3 : (e == 2 ? e_lo : 0)) : 24));
}
constexpr int kCountChoices = 28;           // with padding

struct Plan {
    uint32_t dim[4];              // I, K, L, J of one instance
    uint32_t ndiv[4];
    uint32_t ndiv_inv[4];         // ceil(2^32 / ndiv), for quotients by ndiv of numbers below 2^24 (0 when ndiv is 1)
    uint32_t mirrored;            // bit d: the divisor list of dimension d holds all divisors: cofactors in descending order
    uint32_t instances, n_arrays;
    uint32_t n_orders;            // orders in the search, in row order
    uint32_t order_id[kMaxOrders];
    uint32_t n_blocks;            // (phi, order) blocks in row order, fused first
    uint32_t n_fused_blocks;
    uint32_t fused_tasks;         // n_fused_blocks * 25
    uint8_t  block_phi[kMaxBlocks];
    uint8_t  block_order_slot[kMaxBlocks];   // position of the block's order in order_id[]
    uint32_t tasks_per_tiling;    // fused_tasks + 5 per unfused block
    uint32_t rows_per_tiling;     // R = 125 * tasks_per_tiling
    uint64_t n_tilings;           // T, at most MMEE_MAX_DIVISORS^4 = 2^24
    uint64_t t_begin, t_end;
    int64_t  cap_words;
    int64_t  c_dram_gb;           // quanta per DRAM word moved (DRAM + buffer side)
    int64_t  c_br;                // quanta per buffer<->PE word (buffer + register file side)
    int64_t  c_mac;               // quanta per MAC (MAC + 3 register-file accesses)
    int64_t  c_sfu;               // quanta per softmax element
    int64_t  cq[5];               // raw quantised energies: dram, gb, rf, mac, sfu
    uint32_t has_rf;
    uint32_t bw, pe_rows, pe_cols;
    uint32_t objective, topk;
    uint32_t row_pruning;
    uint32_t fuse_mask;
    uint32_t sm_mask, n_sm;       // stationary pairs in the space (bit s = 3*sm1+sm2; never 0) and their number
    int64_t  key_cap;             // capped objectives: bound on the other key
    uint32_t rf_tiling;           // register-file-level tiling: the block of each operator's tile is searched
    uint32_t rf_words;            // register-file capacity of one PE in words
    double   quantum_pj;
    QueryTables q;
    OrderInfo order[kMaxOrders];  // by order slot
    alignas(16) uint32_t kept_weights[160];   // row pruning only: the kept rows as CountWeights, four bits each
    uint32_t divs[4][MMEE_MAX_DIVISORS];
};

// Host planner (mmee_plan.cu).  Fills `plan`; returns an MMEE_* status.
int build_plan(const mmee_workload_t* w, const mmee_arch_t* a, const mmee_objective_t* o, Plan* plan);
void build_query_tables(QueryTables* q);

// Tie-safe symbolic row pruning (mmee_prune.cu): keep[row] = 1 for the rows of a tiling that are evaluated; the number
// of them; the same by classes; and what the search counts with, in plan->kept_weights (a plan with row_pruning).
void row_pruning_keep(const Plan& plan, uint8_t* keep, uint32_t* kept_rows);
int find_kept_masks(const Plan& plan, KeptMasks* masks, uint32_t* kept_rows);
int set_kept_weights(Plan* plan, uint32_t* kept_rows);

}  // namespace mmee

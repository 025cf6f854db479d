// The kernels' host/device arithmetic as plain functions, for checks on the CPU (tests/test_host_math.py).
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

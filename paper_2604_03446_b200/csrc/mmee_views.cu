// Kernels that evaluate mappings one by one: the key dump, the group flags and full records of an index range.
#include <cuda_runtime.h>

#include "mmee_block.cuh"
#include "mmee_search.h"

namespace mmee {

namespace {

constexpr int kViewThreads = 256;

// One CTA per block of mappings at a time (a grid-stride loop over the range's blocks): the block's level tables are
// built by 32 threads, then every thread evaluates mappings (rows) from them.
template <int OBJ>
__global__ void __launch_bounds__(kViewThreads) dump_kernel(const __grid_constant__ Plan p, int64_t* __restrict__ out) {
    __shared__ BlockTab bt;
    const Limits lim = {p.cap_words, p.key_cap};
    const uint32_t first = (uint32_t)p.t_begin * p.n_blocks, last = (uint32_t)p.t_end * p.n_blocks;
    const uint64_t origin = p.t_begin * p.rows_per_tiling * 9u;
    for (uint32_t id = first + blockIdx.x; id < last; id += gridDim.x) {
        if (threadIdx.x < kBlockItems) block_item(p, PlanDivisors{p}, id, (int)threadIdx.x, &bt);
        __syncthreads();
        const uint32_t n = block_rows(bt) * 9u;
        int64_t* o = out + (bt.first_idx - origin);
        for (uint32_t i = threadIdx.x; i < n; i += kViewThreads) {
            const uint32_t row = i / 9u, s = i - row * 9u;
            const RowTerms r = block_row(p, lim, bt, row);
            o[i] = r.fits && ((p.sm_mask >> s) & 1u) ? mapping_key<OBJ>(p, lim, bt, r, (int)s) : kInfKey;
        }
        __syncthreads();
    }
}

template <int OBJ>
__global__ void __launch_bounds__(kViewThreads) flags_kernel(const __grid_constant__ Plan p, int64_t threshold,
                                                             unsigned char* __restrict__ flags) {
    __shared__ BlockTab bt;
    const Limits lim = {p.cap_words, p.key_cap};
    const uint32_t first = (uint32_t)p.t_begin * p.n_blocks, last = (uint32_t)p.t_end * p.n_blocks;
    const uint64_t origin = p.t_begin * p.rows_per_tiling * 9u;
    for (uint32_t id = first + blockIdx.x; id < last; id += gridDim.x) {
        if (threadIdx.x < kBlockItems) block_item(p, PlanDivisors{p}, id, (int)threadIdx.x, &bt);
        __syncthreads();
        unsigned char* o = flags + (bt.first_idx - origin) / 45u;
        for (uint32_t i = threadIdx.x; i < block_rows(bt) / 5u; i += kViewThreads) {
            bool below = false;
            for (uint32_t e = 0; e < 5; ++e) {
                const RowTerms r = block_row(p, lim, bt, i * 5u + e);
                for (int s = 0; s < 9; ++s)
                    below |= r.fits && ((p.sm_mask >> s) & 1u) && mapping_key<OBJ>(p, lim, bt, r, s) < threshold;
            }
            o[i] = below ? 1 : 0;
        }
        __syncthreads();
    }
}

__global__ void eval_kernel(const __grid_constant__ Plan p, uint64_t idx_begin, uint64_t count,
                            mmee_result_t* __restrict__ out) {
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < count;
         i += (uint64_t)gridDim.x * blockDim.x) {
        mmee_result_t r;
        evaluate_candidate(p, idx_begin + i, r);
        out[i] = r;
    }
}

int block_grid(const Plan& p) {
    const uint64_t n = (p.t_end - p.t_begin) * p.n_blocks;
    return (int)(n < 2368 ? n : 2368);        // 148 SMs x 16 (any number is correct)
}

}  // namespace

cudaError_t launch_dump_keys(const Plan& p, int64_t* out, cudaStream_t st) {
    const int grid = block_grid(p);
    if (!grid) return cudaSuccess;
    switch (p.objective) {
        case MMEE_OBJ_ENERGY: dump_kernel<MMEE_OBJ_ENERGY><<<grid, kViewThreads, 0, st>>>(p, out); break;
        case MMEE_OBJ_LATENCY: dump_kernel<MMEE_OBJ_LATENCY><<<grid, kViewThreads, 0, st>>>(p, out); break;
        case MMEE_OBJ_EDP: dump_kernel<MMEE_OBJ_EDP><<<grid, kViewThreads, 0, st>>>(p, out); break;
        case MMEE_OBJ_ENERGY_LCAP: dump_kernel<MMEE_OBJ_ENERGY_LCAP><<<grid, kViewThreads, 0, st>>>(p, out); break;
        default: dump_kernel<MMEE_OBJ_LATENCY_ECAP><<<grid, kViewThreads, 0, st>>>(p, out); break;
    }
    return cudaGetLastError();
}

cudaError_t launch_group_flags(const Plan& p, int64_t threshold, unsigned char* flags, cudaStream_t st) {
    const int grid = block_grid(p);
    if (!grid) return cudaSuccess;
    switch (p.objective) {
        case MMEE_OBJ_ENERGY: flags_kernel<MMEE_OBJ_ENERGY><<<grid, kViewThreads, 0, st>>>(p, threshold, flags); break;
        case MMEE_OBJ_LATENCY: flags_kernel<MMEE_OBJ_LATENCY><<<grid, kViewThreads, 0, st>>>(p, threshold, flags); break;
        case MMEE_OBJ_EDP: flags_kernel<MMEE_OBJ_EDP><<<grid, kViewThreads, 0, st>>>(p, threshold, flags); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_eval(const Plan& p, uint64_t idx_begin, uint64_t count, mmee_result_t* out, cudaStream_t st) {
    if (!count) return cudaSuccess;
    const uint64_t want = (count + 127) / 128;
    const int grid = (int)(want < 4096 ? want : 4096);
    eval_kernel<<<grid, 128, 0, st>>>(p, idx_begin, count, out);
    return cudaGetLastError();
}

}  // namespace mmee

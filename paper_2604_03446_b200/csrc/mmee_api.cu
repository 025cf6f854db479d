// C ABI of libmmee (declared and documented in include/mmee.h).
#include <cuda_runtime.h>

#include <atomic>
#include <chrono>
#include <cstdlib>
#include <cstring>
#include <new>

#include "mmee_workspace.h"

static_assert(sizeof(mmee_result_t) == 336, "mmee_result_t is part of the ABI");
static_assert(sizeof(mmee::Plan) <= 4096, "the plan travels as a kernel parameter");

struct mmee_handle {
    mmee::Plan plan;
    mmee::LaunchShape shape;
    mmee::Workspace* ws;         // device scratch and pinned host records, from the kept workspaces
    uint32_t kept_rows;          // rows of a tiling that survive pruning (all rows without it)
    int device;
    mmee_launch_stats_t last;
    float create_ms;             // host wall clock of mmee_create
    bool dirty;                  // a launch failed half-way: the scratch header is reset before the next search
    bool in_flight;              // a search was launched whose end this handle has not waited for
    bool timing;
    uint32_t turn;               // searches so far: the last one's scratch is number turn % kScratches
    unsigned long long capture;  // what recorded the last one (capture_of)
    cudaEvent_t ev[2];           // before and after the search kernel
};

namespace {

using namespace mmee;

thread_local cudaError_t g_last_cuda_error = cudaSuccess;

}  // namespace

namespace mmee {

// (An error that is reported here is taken off the runtime, which would otherwise give it to the next launch that asks for
// its last error.)
int cuda_status(cudaError_t e) {
    if (e == cudaSuccess) return MMEE_OK;
    g_last_cuda_error = e;
    cudaGetLastError();
    return MMEE_ERR_CUDA;
}

// Two CTAs per SM (108 to 128 registers a thread, no spills) beat three (80, spilled) and four (64); when the items still counted
// their rows: GQA latency 13.0, 13.7 and 15.1 us, BERT energy 9.4, 10.4 and 12.6, convolution chain top-16 52, 58 and 65.  One slot
// is left free: a search that follows another starts while that one's last CTA finalizes, and a CTA that had to wait for its slot
// would begin its work only then (BERT energy, one search after the other: 16.4 us with all slots taken, 11.6 us with one left; GQA
// latency 20.1 and 13.7).
int max_search_ctas(int device, uint32_t* out) {
    int sm_count = 0;      // attribute query: cudaGetDeviceProperties costs milliseconds
    const cudaError_t e = cudaDeviceGetAttribute(&sm_count, cudaDevAttrMultiProcessorCount, device);
    if (e != cudaSuccess) return cuda_status(e);
    *out = 2u * (uint32_t)sm_count - 1u;
    return MMEE_OK;
}

int choose_launch_shape(const Plan& p, int device, uint32_t n_arrays, uint32_t max_ctas, LaunchShape* shape, uint32_t most) {
    if (!most) {
        const int rc = max_search_ctas(device, &most);
        if (rc) return rc;
    }
    // Small problems take fewer CTAs, with at least eight tilings each.
    const uint64_t tilings = p.t_end - p.t_begin;
    constexpr uint64_t kMinTilings = 8;
    uint64_t grid = (tilings + kMinTilings - 1) / kMinTilings;
    if (grid > most) grid = most;
    if (!grid) grid = 1;
    // (a caller with a fixed scratch: a device that would take more CTAs is refused, not silently under-used)
    if (max_ctas && grid > max_ctas) return MMEE_ERR_RANGE;
    // Passes of equal length, as few as the tables allow.
    const uint64_t per_cta = (tilings + grid - 1) / grid;
    const uint32_t chunk = search_chunk(n_arrays);
    const uint64_t passes = (per_cta + chunk - 1) / chunk;
    shape->grid = (uint32_t)grid;
    shape->n_arrays = n_arrays;
    shape->overlap = true;
    shape->hold = false;
    shape->turn = 0;
    shape->stats = nullptr;
    shape->signal = nullptr;
    shape->signal_value = 0;
    shape->chain_steps = shape->chain_epoch = 0;
    shape->chain_read = false;
    shape->chain_polls = 0;
    shape->chain_to = nullptr;
    shape->chunk = (uint32_t)(passes ? (per_cta + passes - 1) / passes : 1);
    return MMEE_OK;
}

}  // namespace mmee

namespace {

// Waits until a search has written its records, by the word that its last CTA sets in host memory; false: that took longer than a
// short while, and the caller asks the runtime.  The kernel ends a few us later, which a wait for the stream includes, but does
// nothing more to memory: the workspace may be used again.  (One-shot EDP search of 14 336 tilings: 39.6 us with a wait for the
// stream, 37.4 so.  Array shapes, one word for each of eleven: 46.5 and 48.4, so that they wait for the stream.)
bool await_signal(const Workspace* ws) {
    const volatile uint32_t* signal = ws->signal;
    for (uint32_t i = 0; i < 1u << 15; ++i) {
        if (*signal == ws->signals) {
            std::atomic_thread_fence(std::memory_order_acquire);
            return true;
        }
#if defined(__x86_64__)
        __builtin_ia32_pause();
#endif
    }
    return false;
}

// Searches chained on the device (see LaunchShape::chain_steps) until one finds nothing: their optima in order, through
// `take` (which returns false to stop).  The host waits for kHostRecords of them at a time.  Every record a chain may write
// is marked before its launch as one that did not come: whatever its CTAs did not get to shows, MMEE_ERR_TIMEOUT.
template <class Take>
int run_chain(const Plan& plan, uint32_t polls, Take take) {
    int device = 0;
    int rc = cuda_status(cudaGetDevice(&device));
    if (rc) return rc;
    uint32_t most = 0;
    if ((rc = max_search_ctas(device, &most))) return rc;
    most = most + 1 - kChainExtraCtas;      // (all slots: one of them a single search leaves free)
    LaunchShape shape;
    if ((rc = choose_launch_shape(plan, device, 0, 0, &shape, most))) return rc;
    Workspace* ws = nullptr;
    if ((rc = workspace_acquire(device, &ws))) return rc;
    bool more = true, read = false;
    while (more && rc == MMEE_OK) {
        shape.chain_steps = kHostRecords;
        shape.chain_to = ws->chain;
        shape.chain_polls = polls;
        shape.chain_read = read;
        shape.chain_epoch = ++ws->chains * kHostRecords;
        for (uint32_t i = 0; i < kHostRecords; ++i) ws->host[i].status = MMEE_ERR_TIMEOUT;
        const cudaError_t e = launch_search(plan, shape, ws->head, ws->partial[0], nullptr, ws->host_dev, nullptr);
        if (e == cudaErrorCooperativeLaunchTooLarge && shape.grid > 1) {
            // the calling context has a part of the device's SMs: half the CTAs, until they are resident together
            cudaGetLastError();
            rc = choose_launch_shape(plan, device, 0, 0, &shape, shape.grid / 2);
            continue;
        }
        rc = cuda_status(e);
        const int rc2 = cuda_status(cudaStreamSynchronize(nullptr));
        if (rc == MMEE_OK) rc = rc2;
        for (uint32_t i = 0; i < kHostRecords && more && rc == MMEE_OK; ++i) {
            const mmee_result_t& r = ws->host[i];
            if (r.status == MMEE_ERR_CHECK || r.status == MMEE_ERR_TIMEOUT) { rc = r.status; break; }
            more = r.idx != MMEE_NO_INDEX && take(r);
        }
        read = true;
    }
    const int rc2 = workspace_release(ws, rc == MMEE_OK);
    return rc ? rc : rc2;
}

int front_energy_latency(const mmee_workload_t* workload, const mmee_arch_t* arch, const mmee_objective_t* objective,
                         uint32_t polls, mmee_result_t* out_points, uint32_t capacity, uint32_t* n_points) {
    if (!objective || !n_points || (!out_points && capacity)) return MMEE_ERR_ARG;
    *n_points = 0;
    mmee_objective_t o = *objective;
    o.topk = 1; o.row_pruning = 0; o.key_cap = INT64_MAX - 1;
    o.objective = MMEE_OBJ_ENERGY_LCAP;
    Plan plan;
    int rc = build_plan(workload, arch, &o, &plan);
    if (rc) return rc;
    uint32_t n = 0;
    // Each search finds the least energy among the mappings that are still faster than the previous point, and the least
    // latency at that energy: the next point of the front, with its lowest index.  None: the front is complete.
    rc = run_chain(plan, polls, [&](const mmee_result_t& r) {
        if (n < capacity) out_points[n] = r;
        ++n;
        return true;
    });
    *n_points = n;
    if (rc == MMEE_OK && n > capacity) rc = MMEE_ERR_RANGE;
    return rc;
}

int front_buffer_dram(const mmee_workload_t* workload, const mmee_arch_t* arch, const mmee_objective_t* objective,
                      uint32_t polls, mmee_result_t* out_points, uint32_t capacity, uint32_t* n_points) {
    if (!arch || !objective || !n_points || (!out_points && capacity)) return MMEE_ERR_ARG;
    *n_points = 0;
    // DRAM words as the key: one quantum per DRAM word, nothing else costs anything
    mmee_arch_t a = *arch;
    a.e_dram_pj = 1.0; a.e_gb_pj = a.e_rf_pj = a.e_mac_pj = 0.0; a.c_softmax = 0.0; a.energy_quantum_pj = 1.0;
    mmee_objective_t o = *objective;
    o.objective = MMEE_OBJ_ENERGY; o.topk = 1; o.row_pruning = 0; o.key_cap = 0;
    Plan plan;
    int rc = build_plan(workload, &a, &o, &plan);
    if (rc) return rc;
    mmee_result_t held = {};
    bool have = false;
    uint32_t n = 0;
    // Searches with a shrinking buffer: each returns the least DRAM traffic that fits, with the least buffer words that a
    // mapping of the first block with that traffic needs; the next one allows one word less than that.  While the traffic
    // stays the same the mapping found needs less buffer for the same traffic; when it rises, the mapping held is a point
    // of the front.
    auto emit = [&]() {
        if (n < capacity) out_points[n] = held;
        ++n;
    };
    rc = run_chain(plan, polls, [&](const mmee_result_t& r) {
        if (have && r.e_key != held.e_key) emit();
        held = r;
        have = true;
        plan.cap_words = r.bs - 1;      // (for the tables of the next chain: tilings that cannot fit are left out)
        return plan.cap_words >= 0;
    });
    if (rc == MMEE_OK && have) emit();
    // (points whose count of fitting mappings belongs to another bound: see resolve_record)
    mmee_handle_t* h = nullptr;
    for (uint32_t i = 0; i < n && i < capacity && rc == MMEE_OK; ++i) {
        const uint32_t before = out_points[i].reserved2[0];
        if (!before) continue;
        if (!h && (rc = mmee_create(workload, &a, &o, &h))) break;
        h->plan.cap_words = (int64_t)before - 1;
        rc = mmee_search_host(h, &out_points[i], nullptr);
    }
    if (h) {
        const int rc2 = mmee_destroy(h);
        if (rc == MMEE_OK) rc = rc2;
    }
    *n_points = n;
    if (rc == MMEE_OK && n > capacity) rc = MMEE_ERR_RANGE;
    return rc;
}

}  // namespace

extern "C" {

int mmee_create(const mmee_workload_t* workload, const mmee_arch_t* arch, const mmee_objective_t* objective,
                mmee_handle_t** out) {
    if (!out) return MMEE_ERR_ARG;
    *out = nullptr;
    const auto t0 = std::chrono::steady_clock::now();
    mmee_handle* h = new (std::nothrow) mmee_handle;
    if (!h) return MMEE_ERR_ARG;
    std::memset(h, 0, sizeof(*h));
    int rc = build_plan(workload, arch, objective, &h->plan);
    if (rc) { delete h; return rc; }
    if ((rc = cuda_status(cudaGetDevice(&h->device)))) { delete h; return rc; }
    h->kept_rows = h->plan.rows_per_tiling;
    if (h->plan.row_pruning && (rc = set_kept_weights(&h->plan, &h->kept_rows))) { delete h; return rc; }
    rc = choose_launch_shape(h->plan, h->device, 0, 0, &h->shape);
    if (rc) { delete h; return rc; }
    if ((rc = workspace_acquire(h->device, &h->ws))) { delete h; return rc; }
    h->create_ms = std::chrono::duration<float, std::milli>(std::chrono::steady_clock::now() - t0).count();
    *out = h;
    return MMEE_OK;
}

// The handle's device must be the current one: its scratch and tables live there, and a launch from another
// device's context would fail (or, with peer access enabled, silently run on the wrong device).
static int check_device(const mmee_handle* h) {
    int cur = -1;
    const cudaError_t e = cudaGetDevice(&cur);
    if (e != cudaSuccess) return cuda_status(e);
    return cur == h->device ? MMEE_OK : MMEE_ERR_ARG;
}

// The capture that records what is launched on a stream, 0 if there is none.  (The default stream cannot be captured; of one whose
// state is not told the launch will say why, and no search is taken for the one before it.)
static unsigned long long capture_of(cudaStream_t st) {
    if (!st) return 0;
    cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
    unsigned long long number = 0;
    if (cudaStreamGetCaptureInfo(st, &status, &number) != cudaSuccess) {
        cudaGetLastError();
        return UINT64_MAX;
    }
    return status == cudaStreamCaptureStatusNone ? 0 : number | 1ull << 63;
}

// `signalled`: the host will wait for the workspace's signal.
static int search_on(mmee_handle* h, cudaStream_t st, mmee_result_t* out_best, mmee_result_t* out_topk, bool signalled) {
    int rc = check_device(h);
    if (rc) return rc;
    LaunchShape shape = h->shape;
    const unsigned long long capture = capture_of(st);
    if (h->dirty) {        // an earlier launch on this handle failed: a header may hold a used ticket counter
        if ((rc = cuda_status(launch_reset(h->ws->head, st)))) return rc;
        h->dirty = capture != 0;        // (one that is only recorded has not happened)
        shape.overlap = false;          // (its CTAs touch the header: not before the reset has ended)
    }
    // The turns of launched searches and of those that a capture records are one count, but they do not run one after the other:
    // the first after a change of the two (or of captures) starts after what is before it, whose scratches are free then.
    if (capture != h->capture) {
        h->capture = capture;
        shape.overlap = false;
    }
    ++h->turn;
    shape.hold = h->turn % (kScratches - 1) == 0;
    shape.turn = h->turn % kScratches;
    shape.stats = h->ws->stats;
    if (signalled) {
        shape.signal = h->ws->signal_dev;
        shape.signal_value = ++h->ws->signals;
    }
    if (h->timing) cudaEventRecord(h->ev[0], st);
    const cudaError_t e = launch_search(h->plan, shape, h->ws->head, h->ws->partial[shape.turn], out_best, out_topk, st);
    if (e != cudaSuccess) { h->dirty = true; return cuda_status(e); }
    if (h->timing) cudaEventRecord(h->ev[1], st);
    h->last.kernels_launched = 1;
    h->last.grid = h->shape.grid;
    h->last.block = kSearchThreads;
    h->last.smem_bytes = (uint32_t)search_smem_bytes();
    h->last.tasks = (h->plan.t_end - h->plan.t_begin) * h->plan.tasks_per_tiling;
    h->last.rows_per_tiling = h->plan.rows_per_tiling;
    h->last.rows_evaluated_per_tiling = h->kept_rows;
    return MMEE_OK;
}

int mmee_search(mmee_handle_t* h, void* cuda_stream, mmee_result_t* out_best, mmee_result_t* out_topk) {
    if (!h || !out_best) return MMEE_ERR_ARG;
    h->in_flight = true;
    return search_on(h, static_cast<cudaStream_t>(cuda_stream), out_best, out_topk, false);
}

int mmee_search_host(mmee_handle_t* h, mmee_result_t* out_best, mmee_result_t* out_topk) {
    if (!h || !out_best) return MMEE_ERR_ARG;
    const uint32_t k = h->plan.topk;
    int rc;
    // (with timing on, the end of the kernel is wanted and not that of its records)
    if ((rc = search_on(h, nullptr, h->ws->host_dev, h->ws->host_dev + 1, !h->timing))) return rc;
    if ((h->timing || !await_signal(h->ws)) && (rc = cuda_status(cudaStreamSynchronize(nullptr)))) { h->in_flight = true; return rc; }
    std::memcpy(out_best, h->ws->host, sizeof(mmee_result_t));
    if (out_topk) std::memcpy(out_topk, h->ws->host + 1, (size_t)k * sizeof(mmee_result_t));
    return out_best->status == MMEE_ERR_CHECK ? MMEE_ERR_CHECK : MMEE_OK;
}

int mmee_destroy(mmee_handle_t* h) {
    if (!h) return MMEE_ERR_ARG;
    if (h->timing) for (int i = 0; i < 2; ++i) cudaEventDestroy(h->ev[i]);
    int rc = MMEE_OK;
    if (h->in_flight) {
        // A search that the caller launched may still run: the workspace goes to the next handle only after it.  (Its
        // stream may be gone; the wait is the one that freeing device memory implies.)
        int cur = h->device;
        cudaError_t e = cudaGetDevice(&cur);
        if (e == cudaSuccess && cur != h->device) e = cudaSetDevice(h->device);
        if (e == cudaSuccess) e = cudaDeviceSynchronize();
        if (cur != h->device) cudaSetDevice(cur);
        rc = cuda_status(e);
    }
    const int rc2 = workspace_release(h->ws, rc == MMEE_OK && !h->dirty);
    delete h;
    return rc ? rc : rc2;
}

int mmee_trim(void) { return workspace_trim(); }

uint64_t mmee_num_candidates(const mmee_handle_t* h) {
    return h ? h->plan.n_tilings * (uint64_t)h->plan.rows_per_tiling * 9u : 0;
}
uint64_t mmee_num_tilings(const mmee_handle_t* h) { return h ? h->plan.n_tilings : 0; }
uint64_t mmee_num_rows(const mmee_handle_t* h) { return h ? h->plan.rows_per_tiling : 0; }

const char* mmee_strerror(int status) {
    switch (status) {
        case MMEE_OK: return "ok";
        case MMEE_ERR_ARG: return "invalid argument";
        case MMEE_ERR_OVERFLOW: return "a worst-case key of this problem does not fit 62 bits";
        case MMEE_ERR_QUANTUM: return "an energy is not an integer multiple of the energy quantum";
        case MMEE_ERR_NO_FEASIBLE: return "no mapping fits the global buffer";
        case MMEE_ERR_CUDA: return "CUDA runtime error";
        case MMEE_ERR_TIMEOUT: return "device-side wait timed out";
        case MMEE_ERR_RANGE: return "request exceeds a documented maximum";
        case MMEE_ERR_CHECK: return "a winner's ranking key differs from its full evaluation";
        default: return "unknown status";
    }
}

int mmee_eval(mmee_handle_t* h, void* cuda_stream, uint64_t idx_begin, uint64_t count, mmee_result_t* out) {
    if (!h || (!out && count)) return MMEE_ERR_ARG;
    const uint64_t n = mmee_num_candidates(h);
    if (idx_begin > n || count > n - idx_begin) return MMEE_ERR_ARG;
    const int rc = check_device(h);
    if (rc) return rc;
    return cuda_status(launch_eval(h->plan, idx_begin, count, out, static_cast<cudaStream_t>(cuda_stream)));
}

int mmee_decode(mmee_handle_t* h, uint64_t idx, mmee_result_t* host_out) {
    if (!h || !host_out || idx >= mmee_num_candidates(h)) return MMEE_ERR_ARG;
    int rc = check_device(h);
    if (rc) return rc;
    if ((rc = cuda_status(launch_eval(h->plan, idx, 1, h->ws->host_dev, nullptr)))) return rc;
    if ((rc = cuda_status(cudaStreamSynchronize(nullptr)))) { h->in_flight = true; return rc; }
    std::memcpy(host_out, h->ws->host, sizeof(mmee_result_t));
    return MMEE_OK;
}

int mmee_dump_keys(mmee_handle_t* h, void* cuda_stream, int64_t* out_keys) {
    if (!h || !out_keys || h->plan.row_pruning) return MMEE_ERR_ARG;
    const uint64_t n = (h->plan.t_end - h->plan.t_begin) * (uint64_t)h->plan.rows_per_tiling * 9u;
    if (n > (1ull << 31)) return MMEE_ERR_RANGE;
    int rc = check_device(h);
    if (rc) return rc;
    return cuda_status(launch_dump_keys(h->plan, out_keys, static_cast<cudaStream_t>(cuda_stream)));
}

int mmee_filter_flags(mmee_handle_t* h, void* cuda_stream, int64_t threshold_key, uint8_t* out_flags) {
    if (!h || !out_flags || h->plan.row_pruning || h->plan.objective > MMEE_OBJ_EDP) return MMEE_ERR_ARG;
    int rc = check_device(h);
    if (rc) return rc;
    return cuda_status(launch_group_flags(h->plan, threshold_key, out_flags, static_cast<cudaStream_t>(cuda_stream)));
}

int mmee_solve_host(const mmee_workload_t* workload, const mmee_arch_t* arch, const mmee_objective_t* objective,
                    mmee_result_t* out_best, mmee_result_t* out_topk, uint64_t* h2d_bytes, uint64_t* d2h_bytes) {
    if (!out_best || !objective) return MMEE_ERR_ARG;
    mmee_handle_t* h = nullptr;
    int rc = mmee_create(workload, arch, objective, &h);
    if (rc) return rc;
    const uint32_t k = h->plan.topk;
    rc = mmee_search_host(h, out_best, out_topk);
    // The plan (divisor lists, query vectors, coefficients) travels to the device as the search kernel's parameter block,
    // with the launch shape and four pointers: one launch.
    if (h2d_bytes) *h2d_bytes = sizeof(mmee::Plan) + sizeof(mmee::LaunchShape) + 4 * sizeof(void*);
    if (d2h_bytes) *d2h_bytes = sizeof(mmee_result_t) * (uint64_t)(1 + (out_topk ? k : 0));
    const int rc2 = mmee_destroy(h);
    return rc ? rc : rc2;
}

int mmee_pareto_front(const mmee_workload_t* workload, const mmee_arch_t* arch, const mmee_objective_t* objective,
                      mmee_result_t* out_points, uint32_t capacity, uint32_t* n_points) {
    return front_energy_latency(workload, arch, objective, kChainPolls, out_points, capacity, n_points);
}

int mmee_pareto_front_bs_da(const mmee_workload_t* workload, const mmee_arch_t* arch, const mmee_objective_t* objective,
                            mmee_result_t* out_points, uint32_t capacity, uint32_t* n_points) {
    return front_buffer_dram(workload, arch, objective, kChainPolls, out_points, capacity, n_points);
}

int mmee_front_with_polls(int buffer_dram, const mmee_workload_t* workload, const mmee_arch_t* arch,
                          const mmee_objective_t* objective, uint32_t polls, mmee_result_t* out_points, uint32_t capacity,
                          uint32_t* n_points) {
    return (buffer_dram ? front_buffer_dram : front_energy_latency)(workload, arch, objective, polls, out_points, capacity, n_points);
}

int mmee_search_shapes(const mmee_workload_t* workload, const mmee_arch_t* arch, const mmee_objective_t* objective,
                       const uint32_t* shapes, uint32_t n_shapes, mmee_result_t* out_per_shape,
                       uint32_t* out_best_shape) {
    if (!arch || !objective || !shapes || !n_shapes || !out_per_shape || !out_best_shape) return MMEE_ERR_ARG;
    *out_best_shape = UINT32_MAX;
    mmee_objective_t o = *objective;
    o.topk = 1;
    o.row_pruning = 0;
    int device = 0;
    int rc = cuda_status(cudaGetDevice(&device));
    if (rc) return rc;
    Workspace* ws = nullptr;
    bool clean = true;
    bool have = false;
    int64_t best_key = 0;
    for (uint32_t i = 0; i < n_shapes; ++i)
        if (!shapes[2 * i] || !shapes[2 * i + 1]) return MMEE_ERR_ARG;
    // Shapes differ in nothing but the array's rows and columns, so that which rows fit and what they fetch is found once
    // for up to kMaxArrays of them; only the stationary-pair terms and the keys are formed per shape.  (Eleven shapes of
    // the BERT-base chain: one launch per shape 180 us, one launch with a share of the CTAs for each 94 us, this 57 us.)
    mmee_arch_t a = *arch;
    a.pe_rows = shapes[0];
    a.pe_cols = shapes[1];
    Plan plan;
    if ((rc = build_plan(workload, &a, &o, &plan))) return rc;
    if ((rc = workspace_acquire(device, &ws))) return rc;
    for (uint32_t i0 = 0; i0 < n_shapes && rc == MMEE_OK; i0 += kMaxArrays) {
        const uint32_t n = n_shapes - i0 < kMaxArrays ? n_shapes - i0 : kMaxArrays;
        LaunchShape shape;
        if ((rc = choose_launch_shape(plan, device, n, 0, &shape))) break;
        std::memcpy(shape.array, shapes + 2 * i0, n * sizeof(shape.array[0]));
        if ((rc = cuda_status(launch_search_arrays(plan, shape, ws->partial[0], ws->host_dev, nullptr)))) clean = false;
        const int rc2 = cuda_status(cudaStreamSynchronize(nullptr));
        if (rc2) clean = false;
        if (rc == MMEE_OK) rc = rc2;
        if (rc != MMEE_OK) break;
        std::memcpy(out_per_shape + i0, ws->host, n * sizeof(mmee_result_t));
        for (uint32_t i = i0; i < i0 + n; ++i) {
            const mmee_result_t& r = out_per_shape[i];
            if (r.status == MMEE_ERR_CHECK) rc = MMEE_ERR_CHECK;
            if (rc != MMEE_OK || r.idx == MMEE_NO_INDEX) continue;
            // the key the search ordered by: energy, latency, or the bit pattern of the positive EDP product
            int64_t key;
            switch (o.objective) {
                case MMEE_OBJ_ENERGY: case MMEE_OBJ_ENERGY_LCAP: key = r.e_key; break;
                case MMEE_OBJ_LATENCY: case MMEE_OBJ_LATENCY_ECAP: key = r.l_key; break;
                default: std::memcpy(&key, &r.edp_key, sizeof(key)); break;
            }
            if (!have || key < best_key) { have = true; best_key = key; *out_best_shape = i; }
        }
    }
    const int rc2 = workspace_release(ws, clean);
    return rc ? rc : rc2;
}

int mmee_query_vector(uint32_t metric, uint32_t phi, uint32_t pi, uint32_t operand, uint32_t beta,
                      uint32_t recompute, uint8_t out_q[8]) {
    if (!out_q || metric > 1 || phi > 2 || pi > 5 || operand > 4 || beta < 3 || beta > 7 || recompute > 1)
        return MMEE_ERR_ARG;
    QueryTables tables;
    build_query_tables(&tables);
    uint8_t q;
    if (metric == 0) {
        q = tables.bs[pi][operand][beta - 3];
    } else if (phi == 0) {
        if (operand == OP_C) return MMEE_ERR_ARG;
        q = tables.da[pi][operand][beta - 3][recompute];
    } else {
        q = tables.da_unfused[pi][operand][beta - 3];
    }
    for (int d = 0; d < 8; ++d) out_q[d] = (uint8_t)((q >> d) & 1u);
    return MMEE_OK;
}

int mmee_row_pruning_keep(const mmee_objective_t* objective, uint8_t* out_keep, uint32_t capacity,
                          uint32_t* out_rows) {
    if (!objective || !out_keep || !out_rows) return MMEE_ERR_ARG;
    // the row space depends on the objective's order set and fusion modes only: plan a unit workload
    const mmee_workload_t w = {1, 1, 1, 1, 1, 1, 1, 1};
    mmee_arch_t a;
    std::memset(&a, 0, sizeof(a));
    a.pe_rows = a.pe_cols = a.n_arrays = 1;
    a.gb_bytes = 16;
    a.dram_words_per_cycle = 1;
    a.energy_quantum_pj = 1.0;
    mmee_objective_t o = *objective;
    o.topk = 1;
    o.row_pruning = 1;
    o.t_begin = o.t_end = 0;
    Plan plan;
    const int rc = build_plan(&w, &a, &o, &plan);
    if (rc) return rc;
    *out_rows = plan.rows_per_tiling;
    if (capacity < plan.rows_per_tiling) return MMEE_ERR_RANGE;
    uint32_t kept = 0;
    row_pruning_keep(plan, out_keep, &kept);
    return MMEE_OK;
}

int mmee_recompute_flag(uint32_t pi, uint32_t beta_c, uint32_t* out_flag) {
    if (!out_flag || pi > 5 || beta_c < 3 || beta_c > 7) return MMEE_ERR_ARG;
    QueryTables tables;
    build_query_tables(&tables);
    *out_flag = tables.recompute[pi][beta_c - 3];
    return MMEE_OK;
}

int mmee_last_search_stats(const mmee_handle_t* h, mmee_launch_stats_t* out) {
    if (!h || !out) return MMEE_ERR_ARG;
    *out = h->last;
    out->search_ms = out->finalize_ms = -1.0f;
    out->create_ms = h->create_ms;
    out->exact_path_visits = 0;
    out->rows_tested = 0;
    if (h->last.kernels_launched) {
        unsigned long long counters[2] = {0, 0};      // (LaunchShape::stats)
        const int rc = cuda_status(cudaMemcpy(counters, h->ws->stats, sizeof(counters), cudaMemcpyDeviceToHost));
        if (rc) return rc;
        out->exact_path_visits = counters[0];
        out->rows_tested = counters[1];
    }
    if (h->timing && h->last.kernels_launched) {
        const cudaError_t e = cudaEventElapsedTime(&out->search_ms, h->ev[0], h->ev[1]);
        if (e != cudaSuccess) return cuda_status(e);
        out->finalize_ms = 0.0f;        // the finalize step runs inside the search kernel (its last CTA)
    }
    return MMEE_OK;
}

int mmee_kernel_timing(mmee_handle_t* h, int enable) {
    if (!h) return MMEE_ERR_ARG;
    if (enable && !h->timing) {
        for (int i = 0; i < 2; ++i) {
            const int rc = cuda_status(cudaEventCreate(&h->ev[i]));
            if (rc) return rc;
        }
        h->timing = true;
    } else if (!enable && h->timing) {
        for (int i = 0; i < 2; ++i) cudaEventDestroy(h->ev[i]);
        h->timing = false;
    }
    return MMEE_OK;
}

const char* mmee_last_cuda_error(void) { return cudaGetErrorString(g_last_cuda_error); }

int mmee_alu_peak(double out[4]) {
    if (!out) return MMEE_ERR_ARG;
    return cuda_status(measure_alu_peak(out));
}

}  // extern "C"

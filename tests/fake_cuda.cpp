// A stand-in for the CUDA runtime and for the library's kernels: enough of both to run the library's host side (mmee_api,
// mmee_workspace, mmee_plan, mmee_prune) on the CPU and to let single calls fail (tests/test_host_fake_runtime.py).
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdlib>
#include <cstring>
#include <functional>
#include <map>
#include <vector>

#include "../paper_2604_03446_b200/csrc/mmee_workspace.h"

namespace {

struct Allocation { size_t bytes; unsigned long long id; int context; };
std::map<char*, Allocation> g_live;             // what has been allocated and not freed
unsigned long long g_next_id = 1;
int g_context = 1;                              // current context
cudaError_t g_last = cudaSuccess;               // the runtime's last error: kept until it is read
int g_fail_malloc = 0, g_fail_host = 0;         // fail that many calls
int g_bad_pointers = 0;                         // launches and frees that were given memory that is not there
int g_points = 0;                               // optima a chain of searches finds
unsigned g_resident = 1000;                     // CTAs of a chain that can be resident at once
int g_searches = 0;                             // search launches
unsigned g_missing = 0;                         // bit i: the record of its search i is not made
std::map<cudaStream_t, unsigned long long> g_captures;      // streams that are capturing: the capture's number
int g_fail_launch = 0;                          // fail that many search launches
int g_late = 0;                                 // that many searches end only when the host waits for their stream
int g_fail_sync = 0;                            // fail that many waits for a stream
int g_syncs = 0;                                // waits for a stream
struct Launch { unsigned long long capture; int turn, overlap, hold; };       // turn -1: a reset of the header
std::vector<Launch> g_launches;
std::function<void()> g_pending;                // the end of a search that is late

unsigned long long capture_of(cudaStream_t st) {
    auto it = g_captures.find(st);
    return it == g_captures.end() ? 0 : it->second;
}

cudaError_t failed(cudaError_t e) { return g_last = e; }

cudaError_t allocate(void** out, size_t bytes, int* fail) {
    if (*fail > 0) { --*fail; return failed(cudaErrorMemoryAllocation); }
    char* p = static_cast<char*>(std::calloc(1, bytes));
    g_live[p] = {bytes, g_next_id++, g_context};
    *out = p;
    return cudaSuccess;
}

const Allocation* find(const void* ptr) {
    const char* c = static_cast<const char*>(ptr);
    auto it = g_live.upper_bound(const_cast<char*>(c));
    if (it == g_live.begin()) return nullptr;
    --it;
    return c < it->first + it->second.bytes ? &it->second : nullptr;
}

cudaError_t release(void* p) {
    if (!p) return cudaSuccess;
    if (!g_live.erase(static_cast<char*>(p))) { ++g_bad_pointers; return failed(cudaErrorInvalidValue); }
    std::free(p);
    return cudaSuccess;
}

// Device memory of another context is not accessible either.
void touch(const void* p) {
    const Allocation* a = p ? find(p) : nullptr;
    if (p && (!a || a->context != g_context)) ++g_bad_pointers;
}

CUresult fake_pointer_attribute(void* data, CUpointer_attribute which, CUdeviceptr ptr) {
    const Allocation* a = find(reinterpret_cast<void*>(ptr));
    if (!a) return CUDA_ERROR_INVALID_VALUE;
    if (which == CU_POINTER_ATTRIBUTE_BUFFER_ID) *static_cast<unsigned long long*>(data) = a->id;
    else if (which == CU_POINTER_ATTRIBUTE_CONTEXT) *static_cast<CUcontext*>(data) = reinterpret_cast<CUcontext>((size_t)a->context);
    else return CUDA_ERROR_INVALID_VALUE;
    return CUDA_SUCCESS;
}
CUresult fake_current(CUcontext* out) {
    *out = reinterpret_cast<CUcontext>((size_t)g_context);
    return CUDA_SUCCESS;
}

}  // namespace

// ---- controls of the tests
extern "C" {
// The context ends with all its memory; the next one has the same handle (`context` unchanged), as after a device reset.
void fake_device_reset() {
    for (auto& a : g_live) std::free(a.first);
    g_live.clear();
}
void fake_set_context(int c) { g_context = c; }
void fake_fail(int mallocs, int host_allocs) { g_fail_malloc = mallocs; g_fail_host = host_allocs; }
void fake_chain(int points, unsigned missing) { g_points = points; g_missing = missing; }
void fake_resident(unsigned ctas) { g_resident = ctas; }
void fake_capture(void* stream, unsigned long long number) {         // 0: ends
    if (number) g_captures[static_cast<cudaStream_t>(stream)] = number;
    else g_captures.erase(static_cast<cudaStream_t>(stream));
}
void fake_fail_launch(int n) { g_fail_launch = n; }
void fake_late(int searches, int failing_syncs) { g_late = searches; g_fail_sync = failing_syncs; }
int fake_syncs() { return g_syncs; }
// Launch number i of searches and resets; false: there are no more.
int fake_launch(int i, unsigned long long* capture, int* turn, int* overlap, int* hold) {
    if (i >= (int)g_launches.size()) return 0;
    const Launch& l = g_launches[i];
    *capture = l.capture; *turn = l.turn; *overlap = l.overlap; *hold = l.hold;
    return 1;
}
int fake_searches() { return g_searches; }
int fake_plan_bytes() { return (int)sizeof(mmee::Plan); }
int fake_live() { return (int)g_live.size(); }
int fake_bad_pointers() { return g_bad_pointers; }
int fake_last_error() { return (int)g_last; }
}

// ---- the runtime
extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) {
    ++g_syncs;
    if (g_fail_sync > 0) { --g_fail_sync; return failed(cudaErrorLaunchFailure); }
    if (g_pending) g_pending();
    g_pending = nullptr;
    return cudaSuccess;
}
cudaError_t cudaStreamGetCaptureInfo(cudaStream_t st, cudaStreamCaptureStatus* status, unsigned long long* number, cudaGraph_t*,
                                     const cudaGraphNode_t**, size_t*) {
    const unsigned long long n = capture_of(st);
    *status = n ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    if (n) *number = n;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 148; return cudaSuccess; }
cudaError_t cudaGetLastError() { const cudaError_t e = g_last; g_last = cudaSuccess; return e; }
const char* cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "no error" : "an error"; }
cudaError_t cudaMalloc(void** p, size_t bytes) { return allocate(p, bytes, &g_fail_malloc); }
cudaError_t cudaFree(void* p) { return release(p); }
cudaError_t cudaHostAlloc(void** p, size_t bytes, unsigned) { return allocate(p, bytes, &g_fail_host); }
cudaError_t cudaFreeHost(void* p) { return release(p); }
cudaError_t cudaHostGetDevicePointer(void** d, void* h, unsigned) { *d = h; return cudaSuccess; }
cudaError_t cudaMemcpy(void* to, const void* from, size_t n, cudaMemcpyKind) { std::memcpy(to, from, n); return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t*) { return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float*, cudaEvent_t, cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaGetDriverEntryPoint(const char* name, void** f, unsigned long long, cudaDriverEntryPointQueryResult* r) {
    *f = !std::strcmp(name, "cuPointerGetAttribute") ? reinterpret_cast<void*>(fake_pointer_attribute)
         : !std::strcmp(name, "cuCtxGetCurrent")     ? reinterpret_cast<void*>(fake_current) : nullptr;
    if (r) *r = *f ? cudaDriverEntryPointSuccess : cudaDriverEntryPointSymbolNotFound;
    return cudaSuccess;
}
}

// ---- the kernels: a search finds mapping 7 of tiling 0; a launch reports the runtime's last error
namespace mmee {

size_t search_smem_bytes() { return 0; }
uint32_t search_chunk(uint32_t) { return kMaxChunk; }

static mmee_result_t found() {
    mmee_result_t r = {};
    r.idx = 7;
    return r;
}

cudaError_t launch_search(const Plan& p, const LaunchShape& shape, SearchHeader* head, Partial* partials, mmee_result_t* best,
                          mmee_result_t* topk, cudaStream_t st) {
    ++g_searches;
    touch(head);
    touch(partials);
    if (g_fail_launch > 0) { --g_fail_launch; return failed(cudaErrorLaunchOutOfResources); }
    g_launches.push_back({capture_of(st), (int)shape.turn, shape.overlap, shape.hold});
    if (shape.chain_steps && shape.grid + kChainExtraCtas > g_resident) return failed(cudaErrorCooperativeLaunchTooLarge);
    if (shape.chain_steps && (uint64_t)shape.chunk > kMaxChunk) ++g_bad_pointers;
    for (int i = 0; i < (int)shape.chain_steps; ++i) {
        mmee_result_t r = found();
        r.e_key = i;
        r.bs = 1000 - i;
        if (i >= g_points) { r.idx = MMEE_NO_INDEX; r.status = MMEE_ERR_NO_FEASIBLE; }
        if (!(g_missing >> i & 1u)) topk[i] = r;
        if (i >= g_points) return cudaSuccess;
    }
    auto end = [k = p.topk, shape, best, topk] {
        if (find(best)) *best = found();
        for (uint32_t i = 0; topk && find(topk) && i < k; ++i) topk[i] = found();
        touch(shape.signal);
        if (shape.signal && find(shape.signal)) *shape.signal = shape.signal_value;
    };
    if (g_late > 0) {
        --g_late;
        g_pending = end;
    } else {
        end();
    }
    return cudaSuccess;
}
cudaError_t launch_search_arrays(const Plan&, const LaunchShape& shape, Partial* partials, mmee_result_t* out, cudaStream_t) {
    touch(partials);
    for (uint32_t i = 0; i < shape.n_arrays; ++i) out[i] = found();
    return cudaSuccess;
}
cudaError_t launch_reset(SearchHeader* head, cudaStream_t st) {
    touch(head);
    g_launches.push_back({capture_of(st), -1, 0, 0});
    return cudaGetLastError();
}
cudaError_t launch_dump_keys(const Plan&, int64_t*, cudaStream_t) { return cudaGetLastError(); }
cudaError_t launch_group_flags(const Plan&, int64_t, unsigned char*, cudaStream_t) { return cudaGetLastError(); }
cudaError_t launch_eval(const Plan&, uint64_t, uint64_t, mmee_result_t* out, cudaStream_t) {
    if (find(out)) *out = found();
    return cudaGetLastError();
}
cudaError_t measure_alu_peak(double*) { return cudaSuccess; }

}  // namespace mmee

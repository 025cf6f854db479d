// Workspaces kept between handles.
//
// A one-shot search takes 20 to 30 us on the device, but cudaMalloc and cudaFree of its scratch took about 700 us of
// host time around it: with no other allocation of the library alive the driver maps and unmaps a 2 MB slab each time
// (a search of 768 tilings through mmee_solve_host: 730 us).  So a workspace that is no longer in use stays in a list,
// at most kMaxIdle of them (0.32 MB of device and 11 KB of pinned host memory each), for the next handle on its device.
// A workspace belongs to one handle or call at a time, whatever thread or stream uses it; mmee_trim frees the idle ones.
// Its memory belongs to the context it was allocated in and ends with it (cudaDeviceReset, a destroyed driver context), so a
// kept one is taken, or freed, only after the driver has confirmed that its allocation is still that one.
#include "mmee_workspace.h"

#include <cuda.h>

#include <mutex>
#include <new>

namespace mmee {

namespace {

constexpr int kMaxIdle = 8;

std::mutex g_mutex;
Workspace* g_idle = nullptr;
int g_n_idle = 0;

// Driver calls, looked up through the runtime so that the library links no driver library; null where there is none.
struct Driver {
    CUresult (*pointer_attribute)(void*, CUpointer_attribute, CUdeviceptr) = nullptr;
    CUresult (*current_context)(CUcontext*) = nullptr;

    Driver() {
        cudaDriverEntryPointQueryResult found;
        void *a = nullptr, *b = nullptr;
        if (cudaGetDriverEntryPoint("cuPointerGetAttribute", &a, cudaEnableDefault, &found) != cudaSuccess ||
            cudaGetDriverEntryPoint("cuCtxGetCurrent", &b, cudaEnableDefault, &found) != cudaSuccess || !a || !b) {
            cudaGetLastError();
            return;
        }
        pointer_attribute = reinterpret_cast<decltype(pointer_attribute)>(a);
        current_context = reinterpret_cast<decltype(current_context)>(b);
    }
};

const Driver& driver() {
    static const Driver d;
    return d;
}

// The driver's number of a device allocation, 0 if it is none (any more).
unsigned long long allocation_id(const void* mem) {
    unsigned long long id = 0;
    const Driver& d = driver();
    if (!d.pointer_attribute || d.pointer_attribute(&id, CU_POINTER_ATTRIBUTE_BUFFER_ID, (CUdeviceptr)mem) != CUDA_SUCCESS) return 0;
    return id;
}

// Whether the workspace's memory still exists; without the driver calls nothing is kept, so that it does.
bool alive(const Workspace* ws) { return !ws->id || allocation_id(ws->chain) == ws->id; }

// The calling thread's context on `device`, its current device.
CUcontext context_on(int device) {
    CUcontext c = nullptr;
    const Driver& d = driver();
    if (!d.current_context) return nullptr;
    if (d.current_context(&c) == CUDA_SUCCESS && c) return c;
    // (a thread that has not called the runtime yet, or a context that was reset: the device's primary one)
    if (cudaSetDevice(device) != cudaSuccess || d.current_context(&c) != CUDA_SUCCESS) return nullptr;
    return c;
}

bool in_context(const Workspace* ws, CUcontext c) {
    CUcontext own = nullptr;
    return c && driver().pointer_attribute(&own, CU_POINTER_ATTRIBUTE_CONTEXT, (CUdeviceptr)ws->chain) == CUDA_SUCCESS && own == c;
}

int free_workspace(Workspace* ws) {
    if (ws->chain && !alive(ws)) {      // gone with its context, the pinned memory as well
        delete ws;
        return MMEE_OK;
    }
    cudaError_t e = ws->chain ? cudaFree(ws->chain) : cudaSuccess;
    if (ws->host) {
        const cudaError_t e2 = cudaFreeHost(ws->host);
        if (e == cudaSuccess) e = e2;
    }
    delete ws;
    return cuda_status(e);
}

int make_workspace(int device, Workspace** out) {
    Workspace* ws = new (std::nothrow) Workspace();
    if (!ws) return MMEE_ERR_ARG;
    ws->device = device;
    int rc = max_search_ctas(device, &ws->max_ctas);
    if (rc) { delete ws; return rc; }
    // one allocation: the chained searches' optima, the header, the counters, then the partial lists
    static_assert(sizeof(ChainRecord) == 48, "a multiple of 16 bytes keeps the rest aligned");
    const size_t chain = kHostRecords * sizeof(ChainRecord), bytes = ws->max_ctas * sizeof(Partial), before = chain + sizeof(SearchHeader) + 16;
    unsigned char* mem = nullptr;
    cudaError_t e = cudaMalloc(reinterpret_cast<void**>(&mem), before + kScratches * bytes);
    ws->chain = reinterpret_cast<ChainRecord*>(mem);
    if (e == cudaSuccess) ws->id = allocation_id(mem);
    if (e == cudaSuccess) {
        ws->head = reinterpret_cast<SearchHeader*>(mem + chain);
        ws->stats = reinterpret_cast<unsigned long long*>(mem + chain + sizeof(SearchHeader));
        for (int i = 0; i < kScratches; ++i) ws->partial[i] = reinterpret_cast<Partial*>(mem + before + i * bytes);
    }
    // portable: usable from every device's context, mapped: kernels write their records straight into it, so that the
    // host needs no copy call after a search, only the synchronisation
    if (e == cudaSuccess)
        e = cudaHostAlloc(reinterpret_cast<void**>(&ws->host), kHostRecords * sizeof(mmee_result_t) + sizeof(uint32_t),
                          cudaHostAllocMapped | cudaHostAllocPortable);
    if (e == cudaSuccess) e = cudaHostGetDevicePointer(reinterpret_cast<void**>(&ws->host_dev), ws->host, 0);
    if (e == cudaSuccess) {
        ws->signal = reinterpret_cast<uint32_t*>(ws->host + kHostRecords);
        ws->signal_dev = reinterpret_cast<uint32_t*>(ws->host_dev + kHostRecords);
        *ws->signal = 0;
    }
    if (e == cudaSuccess) e = launch_reset(ws->head, 0);
    if (e == cudaSuccess) e = cudaStreamSynchronize(0);
    if (e != cudaSuccess) {
        free_workspace(ws);
        return cuda_status(e);
    }
    *out = ws;
    return MMEE_OK;
}

}  // namespace

int workspace_acquire(int device, Workspace** out) {
    {
        std::lock_guard<std::mutex> lock(g_mutex);
        const CUcontext context = g_idle ? context_on(device) : nullptr;
        for (Workspace** at = &g_idle; *at;) {
            Workspace* ws = *at;
            const bool gone = !alive(ws);
            if (gone || (ws->device == device && in_context(ws, context))) {
                *at = ws->next;
                --g_n_idle;
                if (!gone) {
                    *out = ws;
                    return MMEE_OK;
                }
                delete ws;
            } else {
                at = &ws->next;
            }
        }
    }
    const int rc = make_workspace(device, out);
    if (rc != MMEE_ERR_CUDA) return rc;
    workspace_trim();           // (another device's idle workspaces hold pinned host memory)
    return make_workspace(device, out);
}

int workspace_release(Workspace* ws, bool clean) {
    if (clean && ws->id) {
        std::lock_guard<std::mutex> lock(g_mutex);
        if (g_n_idle < kMaxIdle) {
            ws->next = g_idle;
            g_idle = ws;
            ++g_n_idle;
            return MMEE_OK;
        }
    }
    return free_workspace(ws);
}

int workspace_trim() {
    Workspace* list;
    {
        std::lock_guard<std::mutex> lock(g_mutex);
        list = g_idle;
        g_idle = nullptr;
        g_n_idle = 0;
    }
    int rc = MMEE_OK;
    while (list) {
        Workspace* ws = list;
        list = list->next;
        const int r = free_workspace(ws);
        if (rc == MMEE_OK) rc = r;
    }
    return rc;
}

}  // namespace mmee

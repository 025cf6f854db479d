// Internal: the memory a search needs -- device scratch and pinned host records -- kept between handles.
#pragma once

#include "mmee_search.h"

namespace mmee {

// One search's workspace.  Everything a search on the device needs fits it, whatever the problem.
struct Workspace {
    int device;
    unsigned long long id;          // the device allocation's number: the driver gives no other allocation the same one
    SearchHeader* head;             // device; clean while the workspace is not in use
    Partial* partial[kScratches];   // device: the scratches' partial lists
    unsigned long long* stats;      // device, LaunchShape::stats
    uint32_t max_ctas;              // partial lists a scratch has room for
    ChainRecord* chain;             // device, kHostRecords: what chained searches left
    uint32_t chains;                // launches of them
    mmee_result_t* host;            // pinned host memory: kHostRecords records that kernels write into
    mmee_result_t* host_dev;        // the same memory as the device addresses it
    uint32_t *signal, *signal_dev;  // a word behind the records (LaunchShape::signal)
    uint32_t signals;               // the last value that was waited for
    Workspace* next;
};

constexpr uint32_t kHostRecords = 2 * MMEE_MAX_TOPK;
static_assert(kMaxArrays <= kHostRecords, "one record per array shape");

// A workspace on the current device (`device`), for the caller alone until it is given back.
int workspace_acquire(int device, Workspace** out);
// Gives it back.  `clean`: no work on it is in flight and its header is in its initial state; otherwise it is freed.
// Returns the status of the free.
int workspace_release(Workspace* ws, bool clean);
// Frees every workspace that is not in use.
int workspace_trim();

}  // namespace mmee

// The Pareto fronts (0: energy-latency, 1: buffer size / DRAM traffic) with a limit of their own on the waits between their
// searches, LaunchShape::chain_polls: 0 lets every wait run out.  For tests; not part of the ABI.
extern "C" int mmee_front_with_polls(int buffer_dram, const mmee_workload_t* workload, const mmee_arch_t* arch,
                                     const mmee_objective_t* objective, uint32_t polls, mmee_result_t* out_points,
                                     uint32_t capacity, uint32_t* n_points);

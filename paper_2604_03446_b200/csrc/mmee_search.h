// Internal: device scratch layout and kernel launchers (mmee_search.cu, mmee_views.cu), used by the C ABI.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>

#include "mmee_plan.h"

namespace mmee {

constexpr int kSearchThreads = 256;
constexpr uint32_t kMaxChunk = 144;     // tilings whose tables a CTA holds at once

// One CTA's contribution: its k best blocks as (least key, block number) pairs, best first, and its counts.
struct alignas(16) Partial {
    longlong2 e[MMEE_MAX_TOPK];     // x = key, y = block number: one 16-byte word per pair, stored and loaded whole
    uint32_t count;
    uint32_t live_tilings;
    uint64_t feasible_rows;
};

// Scratches of a handle, taken in turn: all but every (kScratches - 1)-th of its searches let the next one start at once (see
// mmee_search.cu), so that more of them overlap with more scratches, at 80 KB of device memory each.  One search after the other,
// with 2, 3, 4 and 6: BERT 9.5, 8.8, 8.4 and 8.2 us, GQA latency 10.9, 10.2, 9.95 and 9.7, convolution chain top-16 33.0, 31.1, 29.9
// and 29.3.
constexpr int kScratches = 4;

// What the CTAs of one search share, for every scratch: the bound (k > 1) and the ticket counter, reset by the finalize step.
struct SearchHeader {
    long long bound[kScratches];            // k > 1: upper bound on the k-th smallest key
    unsigned int done_ctas[kScratches];     // ticket counter: the CTA that draws the last ticket runs the finalize step
    long long chain_bound;                  // what a chained search leaves to the next one
    unsigned long long chain_epoch;         // the last chained search that has ended on this header (high half)
};
static_assert(sizeof(SearchHeader) == 64, "the header is 64 bytes");

// Global scratch of one search after the other: a header and one partial list per CTA.
struct Scratch {
    SearchHeader head;
    Partial partial[1];     // grid entries follow
};

constexpr uint32_t kMaxArrays = MMEE_MAX_TOPK;      // one entry of a partial list each

// What a chained search leaves of its optimum: key kInfKey if nothing fits; an energy search its key, the block, the buffer
// words it was found under and the least need of a mapping of the block with that key; a search of the energy-latency
// front the latency, the block and the energy.
struct ChainRecord {
    long long key;
    unsigned long long where;
    unsigned long long n_feasible;
    long long bound;
    long long need, pad;
};

struct LaunchShape {
    uint32_t grid;          // CTAs; CTA c takes one tiling of every `grid` consecutive ones
    uint32_t chunk;         // tilings a CTA evaluates per pass, at most kMaxChunk
    uint32_t n_arrays;      // logical array shapes searched by one launch, 0: the plan's own
    uint32_t array[kMaxArrays][2];      // their PE rows and columns
    uint32_t turn;          // the scratch: which entries of the header
    unsigned long long* stats;          // device, 2: groups of 45 mappings of the winning blocks, evaluated one by one; different
                                        // rows of the tilings that were evaluated (null: not wanted)
    uint32_t* signal;       // pinned host memory as the device addresses it: `signal_value` goes there when the records are written (null:
    uint32_t signal_value;  // nobody waits for it)
    bool overlap;           // may start before the kernel before it on the stream has ended (see mmee_search.cu)
    bool hold;              // ... and lets the one after it start only then
    uint32_t chain_steps;   // a chain of this many searches in one launch, 0: one search
    uint32_t chain_epoch;   // ... their numbers on this scratch, ascending and greater than any before: the first one's
    bool chain_read;        // ... that goes on from the launch before
    uint32_t chain_polls;   // ... how often a CTA looks for the end of a search before it gives up (see kChainPolls)
    ChainRecord* chain_to;  // device: where they leave their optima
};
// Chained searches (k = 1, no row pruning; the Pareto fronts): each takes a bound from what the one before it found: the
// buffer words (energy) or the bound on the latency (energy under a latency bound: then the least latency at the least
// energy), not above the plan's.  They are the steps of one kernel, so that the host waits once for all and the tilings'
// tables stay in shared memory; after one that found nothing the chain ends.  A chained search leaves no record but a
// ChainRecord: the next one has to wait for it, and the records are made by
// kRecordCtas more while the searches go on (in out_topk).  (A record takes longer than a short search.  Front of the GPT-3 FFN:
// one 217 us, two 202, four 205 because the searches have fewer CTAs; records after the chain 204, where a front of one point
// takes 59 instead of 55.)
constexpr uint32_t kRecordCtas = 2;
// CTAs of a chain beside those that search: they make the records, and one merges what the others publish.
constexpr uint32_t kChainExtraCtas = kRecordCtas + 1;
// The wait for a chained search is limited, at a few seconds.  A CTA whose wait runs out leaves without a trace: it takes no
// part in later searches, which then do not end, and makes no more records, so that the caller finds one that was not made.
constexpr uint32_t kChainPolls = 1u << 22;

size_t search_smem_bytes();
// Tilings whose tables a CTA holds at once, with the stationary-pair terms of n_arrays array shapes.
uint32_t search_chunk(uint32_t n_arrays);
// One launch per search: the last CTA to finish merges the partial lists, evaluates the winners' blocks mapping by
// mapping, writes the records to out_best / out_topk (device) and resets the scratch header.
cudaError_t launch_search(const Plan& p, const LaunchShape& shape, SearchHeader* head, Partial* partials,
                          mmee_result_t* out_best, mmee_result_t* out_topk, cudaStream_t st);
// The same search (k = 1) on each of shape.n_arrays logical arrays, one record each in `out`: two launches.
cudaError_t launch_search_arrays(const Plan& p, const LaunchShape& shape, Partial* partials, mmee_result_t* out, cudaStream_t st);
cudaError_t launch_reset(SearchHeader* head, cudaStream_t st);

// Every key of the plan's tiling range (kInfKey where a mapping does not fit or its stationary pair is not offered).
cudaError_t launch_dump_keys(const Plan& p, int64_t* out, cudaStream_t st);
// One byte per group of 45 mappings of the range: 1 if one that fits has a key below `threshold`.
cudaError_t launch_group_flags(const Plan& p, int64_t threshold, unsigned char* flags, cudaStream_t st);
cudaError_t launch_eval(const Plan& p, uint64_t idx_begin, uint64_t count, mmee_result_t* out, cudaStream_t st);
cudaError_t measure_alu_peak(double* giops);

// Most CTAs that a search on `device` takes.
int max_search_ctas(int device, uint32_t* out);
// Launch shape of a search of n_arrays array shapes (0: the plan's own) on `device` (for a scratch of max_ctas CTAs when that
// is not 0: MMEE_ERR_RANGE if it would take more).  `most`: CTAs it takes at most, when that is not 0.
int choose_launch_shape(const Plan& p, int device, uint32_t n_arrays, uint32_t max_ctas, LaunchShape* shape, uint32_t most = 0);

// MMEE_OK, or MMEE_ERR_CUDA with the error kept for mmee_last_cuda_error (per host thread).
int cuda_status(cudaError_t e);

}  // namespace mmee

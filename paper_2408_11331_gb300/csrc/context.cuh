// Host-side state of a context (cc_ctx) and the internal calls that the
// served form (server.cu) builds on: sizing a set of jobs before creating it,
// creating a context from a memory pool, and running it without blocking.
#pragma once

#include <map>
#include <string>
#include <vector>

#include "cc_internal.cuh"

struct cc_ctx {
    int jobs = 0, kmax = 0;
    long long n = 0, nnz = 0, rows = 0, keys = 0;
    int device = 0, sms = 0;
    cudaStream_t stream = nullptr;      // stream used by calls
    cudaStream_t own_stream = nullptr;  // stream created by the context (also used for capture)
    cudaStream_t body_stream = nullptr; // captures the bodies of a sweep graph's conditional regions
    cudaStream_t loop_stream = nullptr; // captures the body of its loop
    cudaMemPool_t pool = nullptr;       // device memory comes from this pool (stream-ordered) if set
    std::vector<ccg::JobInfo> job;      // host copy of the job table
    std::vector<long long> psq;         // sum_ij |P_ij|^2 of each job
    std::vector<int> pfirst;            // first global partition of each job
    std::vector<long long> eo;          // first CSR entry of each job (jobs + 1)
    // capacity of each job's place in the union (its sizes at creation): a
    // served context can load a smaller job into a place whose job is done
    std::vector<long long> slot_n, slot_nnz;
    std::vector<int> slot_k;
    std::vector<long long> lbase;       // first label id of each job in a job-concatenated id space
    long long nlabels = 0;              // sum_j k_j 2^s_j
    int parts = 0;                      // sum_j k_j
    long long classes = 0;              // label classes of all partitions (at most)
    int* d_pfirst = nullptr;
    long long* d_lbase = nullptr;
    long long* part_sq = nullptr;       // per global partition: sum_l |P_il|^2
    double* part_slog = nullptr;        // per global partition: sum_l |P_il| log |P_il|
    ccg::JobInfo* d_job = nullptr;
    ccg::JobState* js = nullptr;
    long long* off = nullptr;
    int* col = nullptr;
    int* src = nullptr;
    int* jid = nullptr;
    int* G = nullptr;
    int4* summ = nullptr;
    int* C = nullptr;
    int* size = nullptr;
    int* dsize = nullptr;
    unsigned long long* best = nullptr;
    int4* G16 = nullptr;
    int2* own = nullptr;
    int* chg = nullptr;                 // active set: change stamp per cluster id (n)
    unsigned long long* prev = nullptr; // active set: previous bid per vertex (n)
    unsigned char* act = nullptr;       // active set: scored in this sweep (n)
    ccg::Slot* table = nullptr;
    int* pv = nullptr;
    int* pa = nullptr;
    int* pb = nullptr;
    int* pg = nullptr;
    unsigned char* pflag = nullptr;
    int* members = nullptr;             // rebuild scratch (n)
    int* cursor = nullptr;              // rebuild scratch (n)
    int* bsum = nullptr;                // rebuild scratch (bsum_entries)
    int* scratch = nullptr;             // 3n + n/1024 + 64 ints: output renumbering, warm starts
    // colour_batched: colour of each vertex, vertices and CSR entries by class
    int* colour = nullptr;
    int* vlist = nullptr;
    int* voff = nullptr;
    int* eidx = nullptr;
    long long* eoff = nullptr;
    long long* ccnt = nullptr;          // colouring scratch (2 (n + 2)) and a flag
    int ncls = 1;                       // colour classes (1 without colour_batched)
    bool tuned = true;                  // autotune: lanes chosen (or not to be tuned)
    ccg::DevState* st = nullptr;
    cc_sweep_info* hist = nullptr;
    int hist_cap = 0;
    ccg::SweepArgs args{};
    std::map<int, cudaGraphExec_t> graphs;  // by the number of sweeps in the graph (0: a run's loop)
    std::vector<float> sweep_ms;        // device time of each sweep of the last run
    std::vector<float> propose_ms;      // ... and of its proposal kernels
    long long launches = 0;             // kernels launched so far
    int grid = 0;
    bool run_kernel = false;            // runs go through the run kernel where it can be resident
    int run_blocks = 0;                 // most blocks of the run kernel; 0: runs are graphs of one kernel per step
    int run_want = 0;                   // blocks that the context's work fills
    int in_flight = 0;                  // blocks of its launch of the run kernel that may still run
    unsigned long long* ts = nullptr;   // three device times per sweep body (kRunBodies of them)
    int ts_from = 0, ts_bodies = 0;     // bodies of the last launch not yet in sweep_ms (read when asked for)
    unsigned long long cap_start = 0;   // active table capacity at the singleton start
    unsigned long long cap_max = 0;     // allocated table capacity
    cc_options opt{};
    std::vector<void*> allocs;
    unsigned char* block = nullptr;     // the allocation that holds the context's arrays
    size_t block_bytes = 0, block_used = 0;
    unsigned char* work = nullptr;      // scratch of the distances to the inputs, kept where it is small (in allocs)
    size_t work_bytes = 0;
    size_t bytes = 0;                   // device bytes held
    std::string err;
    // a run driven without blocking (ctx_async_*)
    ccg::DevState* hstate = nullptr;    // pinned host copy of st, owned by the caller
    ccg::JobState* hjobs = nullptr;     // pinned host copy of the job records, owned by the caller (or null)
    cudaEvent_t chunk_done = nullptr;   // recorded after each graph launch and the copy of st
    int async_limit = 0;
    int async_launches = 0;
    bool async_fresh = false;           // the next launch of the run kernel starts the run
};

namespace ccg {

// Entries of the block sums of the run kernel's size scan.
constexpr size_t bsum_entries(size_t n)
{
    return n / 1024 + 4096;
}

// One input job, pointers host or device.
struct JobInput {
    int32_t n;
    int64_t nnz;
    const int64_t* row_off;
    const int32_t* col;
    int32_t k;
    const int32_t* labels;
};

// Sizes of a context for a set of jobs, and the device bytes it holds.
struct Plan {
    int jobs = 0, kmax = 0, hist_cap = 0;
    long long n = 0, nnz = 0, rows = 0, keys = 0, parts = 0, words16 = 0;
    unsigned long long cap_max = 0, cap_start = 0, lcap = 0;
    size_t persistent = 0;  // held until cc_destroy
    size_t temporary = 0;   // held during creation only
};

// Checks the sizes of the jobs and the options (host only; the data pointers
// are not looked at) and sizes the context; *msg gets the reason of a failure.
cc_status plan_jobs(int jobs, const JobInput* in, const cc_options& opt, Plan* out, std::string* msg);
cc_status check_options(const cc_options& opt, std::string* msg);
// Fills the capacities and byte counts of a plan from its totals (jobs, n,
// nnz, rows, words16, keys, parts, kmax).
void finish_plan(Plan& p, const cc_options& opt);
// Lanes that score one (vertex, candidate) pair for partitions of count k.
int lanes_for_k(int k);

// Options with the defaults filled in.
cc_options resolve_options(const cc_options* opt);

// cc_create / cc_batch_create with device memory from `pool` (stream-ordered
// allocation on the context's own stream) when pool is not null; the own
// stream gets the given CUDA stream priority (lower numbers run first).
cc_status ctx_create(int jobs, const JobInput* in, bool on_device, const cc_options* opt, void* stream,
                     cudaMemPool_t pool, cc_ctx** out, int priority = 0);

// Starts a run of at most `limit` sweeps without waiting: queues the run and
// its first launch, then a copy of the control block into `pinned` and an event.
cc_status ctx_async_start(cc_ctx* c, int limit, DevState* pinned, JobState* pinned_jobs = nullptr);

// Checks a run started by ctx_async_start: 0 = its launch still runs, 1 = every job
// has stopped, 2 = the launch ended and the run goes on (the pinned job records
// are those after it: a job with stop set is done and its labels are final;
// ctx_async_continue queues the next launch), -1 = failed (*st holds the status).
int ctx_async_poll_step(cc_ctx* c, cc_status* st);
cc_status ctx_async_continue(cc_ctx* c);
// If the launch has ended, it no longer counts as one that shares the GPU.
void ctx_end_launch(cc_ctx* c);

// Whether a job of these sizes fits the place of job j (see ctx_load_job):
// no more vertices, CSR entries, partitions, label rows or keys than the
// place, and at least a quarter of its vertices and CSR entries.
bool ctx_slot_fits(const cc_ctx* c, int j, const JobInput& in);

// Loads a new job into the place of job j, whose run has ended and whose
// results were taken, while the context's other jobs keep running: the CSR,
// the compacted labels and the singleton state of the new job go into job
// j's ranges (vertices the new job does not use go to an idle job that
// never runs; CSR entries it does not use become self-loops of its last
// vertex, which the method ignores), job j's record restarts at the new
// job's singleton start, the finished job's contingency keys get count 0
// and the new job's singleton keys are inserted (only if the table runs
// short is it rebuilt from C, in the next sweep).  The new job's results are
// then those of running it alone.  Host inputs are read before the call returns.  The run goes on
// with ctx_async_continue.  Errors: CC_ERR_INVALID (malformed input; the
// context is unchanged), CC_ERR_OOM, CC_ERR_CUDA.
cc_status ctx_load_job(cc_ctx* c, int j, const JobInput& in);

// Labels of job j alone, renumbered as by cc_job_labels, into host memory
// (blocks until they are there).  Valid once the job has stopped, also
// while other jobs of the context still run.
cc_status ctx_job_labels_now(cc_ctx* c, int j, int32_t* out);

void ctx_destroy(cc_ctx* c);

}  // namespace ccg

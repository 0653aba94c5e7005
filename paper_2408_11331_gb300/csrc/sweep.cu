// One synchronous local-move sweep (Methods, "Parallel algorithm") of every
// job of a context.  The steps are device functions (sweep_phases.cuh,
// rebuild.cuh); most contexts go through them in the run kernel
// (persist.cu).  Here they are kernels, a fixed sequence on one stream that
// can be captured in a CUDA graph, for small single jobs and for profilers:
//
//   begin        per-sweep counters (union-wide and per job), the sweep's
//                stamp; the sweep is skipped once every job has stopped
//   own/edges/   best move of every vertex against the sweep-start state
//   collect      (Eq. objective4 with the gain of Eq. objective3): what the
//                options need per vertex, then lane groups scoring the
//                distinct candidates of every 128 CSR entries and bidding,
//                then the proposal list
//   route        heavy or light evaluation of the kept moves P1 (results agree)
//   [heavy path] apply P1, rebuild the table (first at a tight capacity, and
//                again at a safe one if the keys did not fit), A_a of every
//                vertex whose cluster changed and with it F' - F per job;
//                commit, or
//   [rollback]   undo and rebuild
//   [light path] singleton guard; stage size and count deltas; exact dF per job
//   bid          matching jobs: drop staged deltas, bid (dD, v) at both clusters
//   match_keys   winners (least (dD, v) at both ends) insert their target keys
//   commit       fold staged deltas in (light P1), move the matching winners;
//                every move stamps its two clusters
//   end          objective, history, stop per job; retry / compaction decisions
//   [rebuild]    rebuild of the contingency hash when one is pending
//
// The bracketed parts are IF regions of the captured graph, entered only when
// a one-thread gate kernel finds them needed (all their kernels also check
// the control block, so a graph without regions gives the same results).
// Entering a region costs 35-43 us and a node 2-5 us, which is why larger
// contexts do not run this way (n = 1e5, k = 8, colour-batched: 15.4 ms as
// graphs, 7.5 ms in the run kernel).
//
// Gain of v moving from its cluster a to b (Eq. objective3, u = v excluded),
// with k the number of partitions of v's job:
//   dD = 2 (A_a - k - A_b) - k (|a| - 1 - |b|),   A_x = sum_i n(x, i, l_i(v)),
// and the move changes the job's F by 2 dD.
#include "sweep_phases.cuh"

namespace ccg {

namespace {

// Entry of the time records for the body that runs now (three words).
__device__ __forceinline__ unsigned long long* body_times(const SweepArgs& a)
{
    return a.ts + 3 * (a.st->run_bodies % kRunBodies);
}

__global__ void k_run_begin(SweepArgs a, int limit, int until)
{
    run_begin_phase(a, limit, until, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}

__global__ void k_run_more(DevState* st, int until)
{
    st->run_until = until;
}

__global__ void k_begin(SweepArgs a)
{
    if (blockIdx.x == 0 && threadIdx.x == 0) body_times(a)[0] = now_ns();
    begin_phase(a, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}

template <bool kSingle>
__global__ void __launch_bounds__(kBlock, 4) k_own(SweepArgs a)
{
    own_phase<kSingle>(a);
}

template <bool kSingle>
__global__ void __launch_bounds__(kBlock, 4) k_edges(SweepArgs a)
{
    __shared__ EdgeScratch sh[kWarpsPerBlock];
    edges_phase<kSingle>(a, sh);
}

__global__ void __launch_bounds__(kBlock) k_collect(SweepArgs a)
{
    collect_phase(a);
}

__global__ void k_route(SweepArgs a)
{
    body_times(a)[1] = now_ns();
    route_phase(a);
}

__global__ void k_h_mark(SweepArgs a)
{
    h_mark_phase(a);
}

__global__ void k_h_apply(SweepArgs a, int undo)
{
    h_apply_phase(a, undo);
}

template <bool kSingle>
__global__ void __launch_bounds__(kBlock, 4) k_h_eval(SweepArgs a)
{
    h_eval_phase<kSingle>(a);
}

__global__ void k_h_decide(SweepArgs a)
{
    h_decide_phase(a, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}

__global__ void k_stage(SweepArgs a)
{
    stage_phase(a);
}

__global__ void k_eval(SweepArgs a)
{
    eval_phase(a);
}

__global__ void k_decide(SweepArgs a)
{
    decide_phase(a, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}

__global__ void k_bid(SweepArgs a)
{
    bid_phase(a);
}

__global__ void k_match_keys(SweepArgs a)
{
    match_keys_phase(a);
}

__global__ void k_commit(SweepArgs a)
{
    commit_phase(a);
}

__global__ void k_match_reset(SweepArgs a)
{
    match_reset_phase(a);
}

__global__ void k_end_jobs(SweepArgs a)
{
    end_jobs_phase(a, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}

__global__ void k_end(SweepArgs a)
{
    if (!a.st->skip) body_times(a)[2] = now_ns();
    end_phase(a);
}

// Regions of a sweep that run only when needed.  In a captured graph each is
// an IF node whose condition a one-thread gate kernel sets from the control
// block, so a sweep that does not need a region skips its launches instead of
// running kernels that return at once.
enum Gate { kGateHeavy = 0, kGateRollback = 1, kGateLight = 2, kGateRebuild = 3, kGateRetry = 4, kGateHeavyEval = 5 };

__global__ void k_gate(cudaGraphConditionalHandle h, DevState* st, int which, int kernels)
{
    const bool run = !st->skip && !st->err;
    bool on = false;
    if (which == kGateHeavy || which == kGateHeavyEval) on = run && st->heavy;
    else if (which == kGateRetry) on = run && st->heavy && st->rebuild;
    else if (which == kGateRollback) on = run && st->heavy && st->rollback;
    else if (which == kGateLight) on = run && !st->heavy && st->nprop > 0;
    else on = st->rebuild && !st->err;
    if (on) st->region_launches += (unsigned long long)kernels;
    cudaGraphSetConditional(h, on ? 1u : 0u);
}

// Opens an IF region in the graph being captured on s: the gate kernel, then
// the conditional node, whose body is captured on b until close_region.
cudaError_t open_region(cudaStream_t s, cudaStream_t b, DevState* st, Gate which, int kernels)
{
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaStreamGetCaptureInfo(s, &cs, nullptr, &g, nullptr, nullptr, nullptr);
    if (e != cudaSuccess) return e;
    if (cs != cudaStreamCaptureStatusActive) return cudaErrorStreamCaptureUnsupported;
    cudaGraphConditionalHandle h = 0;
    e = cudaGraphConditionalHandleCreate(&h, g, 0, 0);
    if (e != cudaSuccess) return e;
    k_gate<<<1, 1, 0, s>>>(h, st, (int)which, kernels);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const cudaGraphNode_t* deps = nullptr;
    const cudaGraphEdgeData* edges = nullptr;
    size_t nd = 0;
    e = cudaStreamGetCaptureInfo(s, &cs, nullptr, &g, &deps, &edges, &nd);
    if (e != cudaSuccess) return e;
    cudaGraphNodeParams p{};
    p.type = cudaGraphNodeTypeConditional;
    p.conditional.handle = h;
    p.conditional.type = cudaGraphCondTypeIf;
    p.conditional.size = 1;
    cudaGraphNode_t node = nullptr;
    e = cudaGraphAddNode(&node, g, deps, edges, nd, &p);
    if (e != cudaSuccess) return e;
    e = cudaStreamUpdateCaptureDependencies(s, &node, nullptr, 1, cudaStreamSetCaptureDependencies);
    if (e != cudaSuccess) return e;
    return cudaStreamBeginCaptureToGraph(b, p.conditional.phGraph_out[0], nullptr, nullptr, 0,
                                         cudaStreamCaptureModeThreadLocal);
}

cudaError_t close_region(cudaStream_t b)
{
    cudaGraph_t g = nullptr;
    return cudaStreamEndCapture(b, &g);
}

// End of one body of a run's loop: go on while the run has not stopped, has no
// error and has bodies left.
__global__ void k_loop_gate(cudaGraphConditionalHandle h, SweepArgs a)
{
    DevState* st = a.st;
    if (st->run_bodies > 0) a.ts[3 * ((st->run_bodies - 1) % kRunBodies) + 2] = now_ns();
    const bool more = !st->stop && !st->err && st->run_bodies < st->run_until;
    cudaGraphSetConditional(h, more ? 1u : 0u);
}

inline int jobs_grid(int jobs)
{
    int g = (jobs + 255) / 256;
    return g < 1 ? 1 : g;
}

}  // namespace

int lanes_for_k(int k)
{
    return lanes_per_item(k);
}

__global__ void k_clear_bids(SweepArgs a)
{
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < a.n; v += stride) a.best[v] = kEmpty;
}

cudaError_t launch_propose_probe(const SweepArgs& a, int grid, cudaStream_t s)
{
    if (a.jobs == 1) {
        k_own<true><<<grid, kBlock, 0, s>>>(a);
        k_edges<true><<<grid, kBlock, 0, s>>>(a);
    } else {
        k_own<false><<<grid, kBlock, 0, s>>>(a);
        k_edges<false><<<grid, kBlock, 0, s>>>(a);
    }
    return cudaGetLastError();
}

cudaError_t launch_clear_bids(const SweepArgs& a, int grid, cudaStream_t s)
{
    k_clear_bids<<<grid, kBlock, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t prepare_propose(int* blocks_per_sm)
{
    int single = 0, multi = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&single, k_edges<true>, kBlock, 0);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&multi, k_edges<false>, kBlock, 0);
    *blocks_per_sm = single < multi ? single : multi;
    return e;
}

cudaError_t capture_run_loop(const SweepArgs& a, long long rows, int grid, cudaStream_t s, cudaStream_t loop,
                             cudaStream_t body)
{
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    cudaGraph_t g = nullptr;
    const cudaGraphNode_t* deps = nullptr;
    const cudaGraphEdgeData* edges = nullptr;
    size_t nd = 0;
    cudaError_t e = cudaStreamGetCaptureInfo(s, &cs, nullptr, &g, &deps, &edges, &nd);
    if (e != cudaSuccess) return e;
    if (cs != cudaStreamCaptureStatusActive) return cudaErrorStreamCaptureUnsupported;
    // the loop is entered once per launch (default value 1); each body's gate
    // decides whether another follows
    cudaGraphConditionalHandle h = 0;
    e = cudaGraphConditionalHandleCreate(&h, g, 1, cudaGraphCondAssignDefault);
    if (e != cudaSuccess) return e;
    cudaGraphNodeParams p{};
    p.type = cudaGraphNodeTypeConditional;
    p.conditional.handle = h;
    p.conditional.type = cudaGraphCondTypeWhile;
    p.conditional.size = 1;
    cudaGraphNode_t node = nullptr;
    e = cudaGraphAddNode(&node, g, deps, edges, nd, &p);
    if (e != cudaSuccess) return e;
    e = cudaStreamUpdateCaptureDependencies(s, &node, nullptr, 1, cudaStreamSetCaptureDependencies);
    if (e != cudaSuccess) return e;
    e = cudaStreamBeginCaptureToGraph(loop, p.conditional.phGraph_out[0], nullptr, nullptr, 0,
                                      cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return e;
    for (int i = 0; i < kLoopSweeps && e == cudaSuccess; ++i) e = launch_sweep(a, rows, grid, loop, body);
    if (e == cudaSuccess) {
        k_loop_gate<<<1, 1, 0, loop>>>(h, a);
        e = cudaGetLastError();
    }
    cudaGraph_t lg = nullptr;
    const cudaError_t e2 = cudaStreamEndCapture(loop, &lg);
    return e != cudaSuccess ? e : e2;
}

cudaError_t launch_run_begin(const SweepArgs& a, int limit, int until, cudaStream_t s)
{
    k_run_begin<<<jobs_grid(a.jobs), 256, 0, s>>>(a, limit, until);
    return cudaGetLastError();
}

cudaError_t launch_run_more(const SweepArgs& a, int until, cudaStream_t s)
{
    k_run_more<<<1, 1, 0, s>>>(a.st, until);
    return cudaGetLastError();
}

cudaError_t launch_sweep(const SweepArgs& a, long long rows, int grid, cudaStream_t s, cudaStream_t body)
{
    const int g2 = grid;
    const int jg = jobs_grid(a.jobs);
    const size_t js1 = smem_jobs_bytes(a.jobs);
    cudaError_t e = cudaSuccess;
    // with a body stream, the optional regions are IF nodes of the captured
    // graph (their kernels also check the control block themselves)
    auto open = [&](Gate which, int kernels) -> cudaStream_t {
        if (!body || e != cudaSuccess) return s;
        e = open_region(s, body, a.st, which, kernels);
        return body;
    };
    auto close = [&]() {
        if (body && e == cudaSuccess) e = close_region(body);
    };
    k_begin<<<jg, 256, 0, s>>>(a);
    if (a.jobs == 1) {
        k_own<true><<<grid, kBlock, 0, s>>>(a);
        k_edges<true><<<grid, kBlock, 0, s>>>(a);
    } else {
        k_own<false><<<grid, kBlock, 0, s>>>(a);
        k_edges<false><<<grid, kBlock, 0, s>>>(a);
    }
    k_collect<<<grid, kBlock, js1, s>>>(a);
    k_route<<<1, 1, 0, s>>>(a);
    {
        cudaStream_t r = open(kGateHeavy, 2 + kKernelsPerRebuild);
        if (e != cudaSuccess) return e;
        k_h_mark<<<g2, kBlock, js1, r>>>(a);
        k_h_apply<<<g2, kBlock, 0, r>>>(a, 0);
        e = launch_table_rebuild(a, rows, true, r);
        if (e != cudaSuccess) return e;
        close();
        if (e != cudaSuccess) return e;
    }
    {
        // second attempt of the heavy rebuild, when the tight capacity was
        // too small (the rebuild is still pending)
        cudaStream_t r = open(kGateRetry, kKernelsPerRebuild);
        if (e != cudaSuccess) return e;
        e = launch_table_rebuild(a, rows, true, r);
        if (e != cudaSuccess) return e;
        close();
        if (e != cudaSuccess) return e;
    }
    {
        cudaStream_t r = open(kGateHeavyEval, 2);
        if (e != cudaSuccess) return e;
        if (a.jobs == 1) k_h_eval<true><<<g2, kBlock, js1, r>>>(a);
        else k_h_eval<false><<<g2, kBlock, js1, r>>>(a);
        k_h_decide<<<jg, 256, 0, r>>>(a);
        e = cudaGetLastError();
        close();
        if (e != cudaSuccess) return e;
    }
    {
        cudaStream_t r = open(kGateRollback, 1 + kKernelsPerRebuild);
        if (e != cudaSuccess) return e;
        k_h_apply<<<g2, kBlock, 0, r>>>(a, 1);
        e = launch_table_rebuild(a, rows, true, r);
        if (e != cudaSuccess) return e;
        close();
        if (e != cudaSuccess) return e;
    }
    {
        cudaStream_t r = open(kGateLight, 3);
        if (e != cudaSuccess) return e;
        k_stage<<<g2, kBlock, js1, r>>>(a);
        k_eval<<<g2, kBlock, js1, r>>>(a);
        k_decide<<<jg, 256, 0, r>>>(a);
        e = cudaGetLastError();
        close();
        if (e != cudaSuccess) return e;
    }
    k_bid<<<g2, kBlock, 0, s>>>(a);
    k_match_keys<<<g2, kBlock, 0, s>>>(a);
    k_commit<<<g2, kBlock, 2 * a.jobs <= kSmemJobs ? 2 * smem_jobs_bytes(a.jobs) : 0, s>>>(a);
    k_match_reset<<<g2, kBlock, 0, s>>>(a);
    k_end_jobs<<<jg, 256, 0, s>>>(a);
    k_end<<<1, 1, 0, s>>>(a);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    {
        cudaStream_t r = open(kGateRebuild, kKernelsPerRebuild);
        if (e != cudaSuccess) return e;
        e = launch_table_rebuild(a, rows, true, r);
        if (e != cudaSuccess) return e;
        close();
    }
    return e;
}

}  // namespace ccg

// The run kernel: a whole run (or a budget of sweep bodies) of a context in
// one cooperative launch.  Its blocks stay resident and go through the steps
// of a sweep (sweep_phases.cuh, rebuild.cuh) together, with a grid barrier
// where a step needs what other blocks wrote; the last block to arrive takes
// the decisions between two steps (route, guards, end of the sweep) while the
// others wait, so a decision costs no pass of its own.
//
// What bounds it: at small and middle sizes the barriers (3-4 us each with 608
// blocks) and the latency of each step's dependent gathers, at large sizes the
// steps themselves (gathers of label and summary rows).  The same steps as a
// graph of kernels with IF regions spent 2-5 us per node and 35-43 us to enter
// a region, about 110 us per sweep, and 1.0-1.5 ms of host time to capture and
// instantiate the graph of a new context.  Measured, graphs then run kernel:
// LFR-style n = 20011, k = 12, host to host 3.31 -> 1.75 ms; colour-batched
// n = 1e5, k = 8 15.4 -> 7.5 ms; 40 served requests 20.2 -> 17.3 ms.
// Layout: 4 blocks of 256 threads per SM (64 registers), as the scoring step
// wants; the steps that gather in shared memory share one buffer, because
// every further KB came out of the L1 that the other steps read through
// (n = 1e6, k = 20: 8.4 -> 7.5 ms).
#include <algorithm>

#include "rebuild.cuh"
#include "sweep_phases.cuh"

namespace ccg {

namespace {

__device__ __forceinline__ unsigned ld_relaxed(const unsigned* p)
{
    unsigned x;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(x) : "l"(p) : "memory");
    return x;
}

__device__ __forceinline__ unsigned atom_add_acq_rel(unsigned* p, unsigned x)
{
    unsigned old;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(x) : "memory");
    return old;
}

__device__ __forceinline__ void st_release(unsigned* p, unsigned x)
{
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(x) : "memory");
}

// Steps of the run kernel.
enum Step {
    kStart, kOwn, kEdges, kCollect,         // proposal step
    kMark, kApply, kUndo, kHeavyEval,       // heavy path (and its rollback)
    kSizes, kClear, kScatter, kBuild, kTop, // table rebuild
    kStage, kEval,                          // light path
    kBid, kKeys, kCommit,                   // matching, commit
    kBegin, kDecide, kHeavyDecide, kEndJobs, // per-job decisions of many jobs
    kLeave
};

// Up to this many jobs the block that takes the decisions goes through them
// alone, 256 at a time; more are a step of all blocks.  A step costs a barrier
// (three of them per sweep), the rounds of one block 1-2 us each.  Runs, alone
// and as steps: 512 jobs of n = 300 1463 and 1502 us, 1000 of 120 1161 and 1130,
// 8000 of 60 3086 and 2448, 120,000 of 8 9.45 and 3.12 ms.
constexpr int kSchedulerJobs = 768;

// Grid barrier between two steps.  The last block to arrive runs schedule()
// (all its threads; the value counts in thread 0), which takes the decisions
// that follow from the finished step and returns the next one; the others
// wait for it.  Barrier number and next step travel in one word, so every
// block takes the same step without another load.  A wait that exceeds
// wait_ns sets st->err and ends the kernel in every block: the blocks still at
// work finish their step and at most one more, for no later barrier sees all
// of them.
template <class Schedule>
__device__ __forceinline__ int grid_step(DevState* st, unsigned long long wait_ns, unsigned& word, unsigned& arrivals,
                                         Schedule schedule)
{
    __shared__ unsigned s_word;
    __shared__ int s_last;
    __syncthreads();
    arrivals += gridDim.x;
    if (threadIdx.x == 0) s_last = atom_add_acq_rel(&st->bar_count, 1u) == arrivals - 1;
    __syncthreads();
    if (s_last) {
        const int next = schedule();
        __syncthreads();
        if (threadIdx.x == 0) {
            s_word = (((word >> 8) + 1) << 8) | (unsigned)next;
            if (next == kLeave) st->bar_count = 0;
            st_release(&st->bar_word, s_word);
        }
    } else if (threadIdx.x == 0) {
        unsigned long long t0 = 0;
        unsigned now;
        // relaxed polls and one fence at the end: an acquire on every poll
        // would drop the L1 lines of the blocks still at work on this SM
        for (unsigned spins = 1; (now = ld_relaxed(&st->bar_word)) == word; ++spins) {
            __nanosleep(100);
            if ((spins & 1023u) && wait_ns) continue;
            if (t0 == 0) t0 = now_ns();
            if (*reinterpret_cast<volatile int*>(&st->bar_abort) || !wait_ns || now_ns() - t0 > wait_ns) {
                set_err(st, CC_ERR_TIMEOUT);
                st->bar_abort = 1;
                now = kLeave;
                break;
            }
        }
        __threadfence();
        s_word = now;
    }
    __syncthreads();
    word = s_word;
    return (int)(word & 255u);
}

// Sum of x over the block, in every thread.
__device__ __forceinline__ int block_sum(int x)
{
    __shared__ int part[kWarpsPerBlock];
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = x;
    __syncthreads();
    int s = 0;
#pragma unroll
    for (int w = 0; w < kWarpsPerBlock; ++w) s += part[w];
    return s;
}

// Exclusive scan of the cluster sizes into cursor[], first half: each block's
// sum over its own contiguous range of ids.
__device__ __forceinline__ void scan_range(const SweepArgs& a, long long& lo, long long& hi)
{
    const long long per = ((a.n + gridDim.x - 1) / gridDim.x + 3) & ~3LL;
    lo = per * blockIdx.x < a.n ? per * blockIdx.x : a.n;
    hi = lo + per < a.n ? lo + per : a.n;
}

__device__ __forceinline__ void scan_sum_step(const SweepArgs& a)
{
    long long lo, hi;
    scan_range(a, lo, hi);
    int s = 0;
    unsigned long long small = 0;
    for (long long v = lo + threadIdx.x; v < hi; v += kBlock) {
        s += a.size[v];
        small += small_rows(a, v, a.size[v]);
    }
    if (to_size(a.st, 1)) add_small_rows(a.st, small);
    s = block_sum(s);
    if (threadIdx.x == 0) a.bsum[blockIdx.x] = s;
}

// Second half: the sums of the blocks before, then the block's own range in
// tiles of four ids per thread.
__device__ __forceinline__ void scan_write_step(const SweepArgs& a)
{
    __shared__ int wsum[kWarpsPerBlock];
    long long lo, hi;
    scan_range(a, lo, hi);
    int before = 0;
    for (unsigned b = threadIdx.x; b < blockIdx.x; b += kBlock) before += a.bsum[b];
    int run = block_sum(before);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (long long t = lo; t < hi; t += 4 * kBlock) {
        const long long v = t + 4 * threadIdx.x;
        int s[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) s[i] = v + i < hi ? a.size[v + i] : 0;
        const int mine = s[0] + s[1] + s[2] + s[3];
        const int incl = warp_incl_scan(mine, lane);
        __syncthreads();
        if (lane == 31) wsum[w] = incl;
        __syncthreads();
        int x = run + incl - mine, all = 0;
#pragma unroll
        for (int q = 0; q < kWarpsPerBlock; ++q) {
            if (q < w) x += wsum[q];
            all += wsum[q];
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (v + i < hi) a.cursor[v + i] = x;
            x += s[i];
        }
        run += all;
    }
}

// What follows a finished step (all threads of one block; the decisions of the
// one-thread and per-job steps of a sweep are taken here).
template <bool kSingle>
struct Scheduler {
    const SweepArgs& a;

    __device__ bool many_jobs() const { return !kSingle && a.jobs > kSchedulerJobs; }

    // Starts a rebuild: 0 heavy sweep, 1 its rollback, 2 end of the sweep.
    __device__ int rebuild(int kind) const
    {
        if (threadIdx.x == 0) a.st->rebuild_kind = kind;
        return kSizes;
    }

    __device__ int begin() const
    {
        __syncthreads();
        if (a.st->bodies_left <= 0) return kLeave;
        if (many_jobs()) return kBegin;
        begin_phase(a, threadIdx.x, kBlock);
        return begun();
    }

    __device__ int begun() const
    {
        __syncthreads();
        // the own step only serves these options
        return a.st->skip ? kLeave : a.active_set || a.empty_moves ? kOwn : kEdges;
    }

    // Objective, history and stop per job; then the end-of-sweep rebuild or
    // the next sweep.
    __device__ int end() const
    {
        __syncthreads();
        if (many_jobs()) return kEndJobs;
        end_jobs_phase(a, threadIdx.x, kBlock);
        return ended();
    }

    __device__ int ended() const
    {
        __syncthreads();
        if (threadIdx.x == 0) {
            end_phase(a);
            a.st->bodies_left -= 1;
        }
        __syncthreads();
        return a.st->rebuild && !a.st->err ? rebuild(2) : begin();
    }

    __device__ int after_apply() const { return a.st->match ? kBid : end(); }

    __device__ int next(int step) const
    {
        DevState* st = a.st;
        switch (step) {
        case kStart: return begin();
        case kBegin: return begun();
        case kOwn: return kEdges;
        case kEdges: return kCollect;
        case kCollect:
            if (threadIdx.x == 0) {
                route_phase(a);
                st->tries = 0;
            }
            __syncthreads();
            if (st->heavy) return kMark;
            if (st->nprop > 0 && !st->err) return kStage;
            return end();
        case kMark: return kApply;
        case kApply: return rebuild(0);
        case kUndo: return rebuild(1);
        case kSizes:
            if (threadIdx.x == 0 && to_size(st, 1)) size_build(a);
            return kClear;
        case kClear: return kScatter;
        case kScatter: return kBuild;
        case kBuild: build_check_phase(a, 1); return kTop;
        case kTop:
            if (threadIdx.x == 0) {
                table_done_phase(st, 1);
                st->tries += 1;
            }
            __syncthreads();
            if (st->rebuild_kind == 2) return begin();
            if (st->rebuild_kind == 1) return after_apply();
            if (st->again && st->tries < 2) return kSizes;  // the tight attempt did not fit
            return kHeavyEval;
        case kHeavyEval:
            if (many_jobs()) return kHeavyDecide;
            h_decide_phase(a, threadIdx.x, kBlock);
            __syncthreads();
            return st->rollback ? kUndo : after_apply();
        case kHeavyDecide: return st->rollback ? kUndo : after_apply();
        case kStage: return kEval;
        case kEval:
            if (many_jobs()) return kDecide;
            decide_phase(a, threadIdx.x, kBlock);
            __syncthreads();
            return st->match ? kBid : kCommit;
        case kDecide: return st->match ? kBid : kCommit;
        case kBid: return kKeys;
        case kKeys: return kCommit;
        case kCommit: return end();
        case kEndJobs: return ended();
        }
        return kLeave;
    }
};

// The steps below are functions of their own: inlined in the step loop, their
// index arithmetic is hoisted out of it and kept in registers across the other
// steps, which then spill (a run at n = 1e6, k = 20: 7.04 ms inlined, 6.84 so;
// 48 jobs as one batch: 7.69 and 7.54; a k-NN graph, n = 2e6, k = 50: 25.7 and
// 25.4).  All in one function was worse again (light steps +15%).  The scoring,
// the heavy evaluation, the proposal list and the commit stay inlined: they read
// the arguments too often to go through a pointer.
template <bool kSingle>
__device__ __noinline__ void own_step(const SweepArgs& a)
{
    own_phase<kSingle>(a);
}

__device__ __noinline__ void mark_step(const SweepArgs& a)
{
    h_mark_phase(a);
}

__device__ __noinline__ void apply_step(const SweepArgs& a, int undo)
{
    h_apply_phase(a, undo);
}

__device__ __noinline__ void sizes_step(const SweepArgs& a)
{
    scan_sum_step(a);
}

__device__ __noinline__ void clear_step(const SweepArgs& a, long long rows)
{
    table_clear_phase(a, rows, 1);
    scan_write_step(a);
}

__device__ __noinline__ void scatter_step(const SweepArgs& a, TileCount* tc)
{
    members_scatter_phase(a, 1, tc);
}

__device__ __noinline__ void build_step(const SweepArgs& a)
{
    table_build_phase(a, 1);
}

__device__ __noinline__ void top_step(const SweepArgs& a)
{
    summ_top_phase(a, 1);
}

__device__ __noinline__ void stage_step(const SweepArgs& a)
{
    stage_phase(a);
}

__device__ __noinline__ void eval_step(const SweepArgs& a)
{
    eval_phase(a);
}

__device__ __noinline__ void bid_step(const SweepArgs& a)
{
    bid_phase(a);
}

__device__ __noinline__ void keys_step(const SweepArgs& a)
{
    match_keys_phase(a);
}

__device__ __noinline__ void match_reset_step(const SweepArgs& a)
{
    match_reset_phase(a);
}

// The per-job decisions `step` of many jobs, by all blocks.
__device__ __noinline__ void jobs_step(const SweepArgs& a, int step)
{
    const int t0 = blockIdx.x * kBlock + threadIdx.x, stride = gridDim.x * kBlock;
    switch (step) {
    case kBegin: begin_phase(a, t0, stride); break;
    case kDecide: decide_phase(a, t0, stride); break;
    case kHeavyDecide: h_decide_phase(a, t0, stride); break;
    case kEndJobs: end_jobs_phase(a, t0, stride); break;
    }
}

}  // namespace

// fresh: 1 starts a run of at most `limit` sweeps, 0 goes on with it; at most
// `budget` sweep bodies are run.
template <bool kSingle>
__global__ void __launch_bounds__(kBlock, 4)
    k_run(const __grid_constant__ SweepArgs a, long long rows, int limit, int fresh, int budget)
{
    // one buffer for the steps that gather in shared memory, so that the L1
    // keeps the rest
    __shared__ union {
        EdgeScratch edge[kWarpsPerBlock];
        TileCount tile;
    } scratch;
    DevState* st = a.st;
    unsigned arrivals = 0;                       // at the barrier, over this launch
    unsigned word = ld_relaxed(&st->bar_word);   // cannot change before this block arrives
    const bool clock = blockIdx.x == 0 && threadIdx.x == 0;
    int step = kStart, last = kStart, body = -1;
    // every step ends in a barrier; kLeave ends the kernel
    for (;;) {
        if (clock && (step == kOwn || (step == kEdges && last != kOwn))) {
            // a sweep begins
            if (body >= 0) a.ts[3 * body + 2] = now_ns();
            ++body;
            a.ts[3 * body] = now_ns();
        }
        switch (step) {
        case kStart:
            if (clock) st->bodies_left = budget;
            if (fresh) run_begin_phase(a, limit, 0, blockIdx.x * kBlock + threadIdx.x, gridDim.x * kBlock);
            break;
        case kOwn: own_step<kSingle>(a); break;
        case kEdges: edges_phase<kSingle>(a, scratch.edge); break;
        case kCollect: collect_phase(a); break;
        case kMark: mark_step(a); break;
        case kApply: apply_step(a, 0); break;
        case kUndo: apply_step(a, 1); break;
        case kSizes: sizes_step(a); break;
        case kClear: clear_step(a, rows); break;
        case kScatter: scatter_step(a, &scratch.tile); break;
        case kBuild: build_step(a); break;
        case kTop: top_step(a); break;
        case kHeavyEval: h_eval_phase<kSingle>(a); break;
        case kStage: stage_step(a); break;
        case kEval: eval_step(a); break;
        case kBid: bid_step(a); break;
        case kKeys: keys_step(a); break;
        case kCommit:
            commit_phase(a);
            if (st->match) match_reset_step(a);
            break;
        case kBegin:
        case kDecide:
        case kHeavyDecide:
        case kEndJobs:
            if (!kSingle) jobs_step(a, step);
            break;
        }
        const int done = step;
        step = grid_step(st, a.wait_ns, word, arrivals, [&] { return Scheduler<kSingle>{a}.next(done); });
        if (clock && done == kCollect) a.ts[3 * body + 1] = now_ns();
        if (step == kLeave) break;
        last = done;
    }
    if (clock && body >= 0) a.ts[3 * body + 2] = now_ns();
}

namespace {

inline size_t run_smem(int jobs)
{
    return (2 * jobs <= kSmemJobs ? 2 : 1) * smem_jobs_bytes(jobs);
}

// A place for a block that a run leaves free, so that the caller's small kernels
// on other streams find one: four blocks of a run take all registers of an SM,
// and with every place taken such a kernel waited for the end of the run (beside n
// = 300,007, k = 24: one block 1224 us, 48 so; 2^20 floats 1225 and 299; one that
// fills the GPU waits all the same).  It costs a run 0-0.6% (two places 0-6%, where
// a step's rounds of work come out uneven: n = 1e5 with 32 lanes; eight 1%).
inline int spare_blocks(int resident)
{
    return std::min(1, resident / 64);
}

}  // namespace

cudaError_t run_grid(const SweepArgs& a, long long rows, int sms, int* most, int* want)
{
    int per_sm = 0;
    const cudaError_t e =
        a.jobs == 1 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_run<true>, kBlock, run_smem(a.jobs))
                    : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_run<false>, kBlock, run_smem(a.jobs));
    if (e != cudaSuccess) return e;
    long long g = std::max((a.nnz + kBlock - 1) / kBlock, (rows + 8 * kBlock - 1) / (8 * kBlock));
    g = std::max(g, (a.n + kBlock - 1) / kBlock);
    const int resident = per_sm * sms;
    *most = resident - spare_blocks(resident);
    *want = (int)std::min(g, 1LL << 20);
    return cudaSuccess;
}

cudaError_t launch_run(const SweepArgs& a, long long rows, int grid, int limit, bool fresh, int budget, cudaStream_t s)
{
    SweepArgs args = a;
    int f = fresh ? 1 : 0;
    void* params[] = {&args, &rows, &limit, &f, &budget};
    const void* k = a.jobs == 1 ? reinterpret_cast<const void*>(k_run<true>) : reinterpret_cast<const void*>(k_run<false>);
    return cudaLaunchCooperativeKernel(k, dim3((unsigned)grid), dim3(kBlock), params, run_smem(a.jobs), s);
}

}  // namespace ccg

// Internal declarations shared by the CUDA translation units of libcc.so.
//
// A context holds J independent consensus jobs as one disjoint union (a
// single job is J = 1).  Vertices of job j are the union ids vo_j .. vo_j+n_j-1;
// cluster ids are union vertex ids (the founding vertex), so they never clash
// across jobs and a cluster id also names its job.  Every step of a sweep runs
// over the whole union in the same kernels; each job keeps its own counters,
// guard decisions, objective, convergence and history, so a job's run is
// identical to running it alone.
//
// Device data layout:
//   off   int64[N+1]   union CSR row offsets      col  int32[NNZ] union neighbour ids
//   src   int32[NNZ]   source vertex of each CSR entry
//   jid   int32[N]     job of each vertex (and of each cluster id)
//   G     int32[...]   compacted label ids, vertex-major: job j's rows start at go_j,
//                      kp_j = k_j rounded up to 4 ints each (16-byte rows, padding -1);
//                      g = (i << s_j) | rep, rep the job-local index of the least vertex
//                      carrying that label in partition i and 2^s_j >= n_j, so g names
//                      (partition, label) within the job and g < 2 k_j n_j.
//   G16   int4[...]    the same labels as 16-bit class numbers, counted from 0 within each
//                      partition: rows of quads16(k_j) words (valid where JobInfo::narrow)
//   summ  int4[...]    rows as in G, one per cluster id, entries as summ_at places them: per partition i
//                      {d1, m1, d2, m2}: the two label ids that were most frequent in the
//                      cluster at the last table rebuild (d1 first; -1 where the cluster
//                      had fewer labels) and the exact current counts of each (kept by
//                      every commit), so |cluster| - m1 - m2 bounds the count of any
//                      other label (and is 0 when d1 and d2 cover the cluster).  The
//                      first 8 bytes read as one unsigned 64-bit value are m1 << 32 | d1
//                      (likewise the last 8), the order in which the rebuild ranks labels.
//   C     int32[N]     cluster id of each vertex
//   size  int32[N]     cluster sizes, indexed by cluster id
//   table Slot[cap]    the contingency counts n(c, i, l) of all jobs as one open-
//                      addressing hash with linear probing, key = c << 32 | g.  Only an
//                      active prefix of st->mask + 1 slots is used; it is rebuilt from C
//                      (with dead keys dropped) when needed.
#pragma once

#include <cstdint>
#include <string>
#include <vector>
#include <cuda_runtime.h>

#include "cc.h"

namespace ccg {

constexpr unsigned long long kEmpty = ~0ull;
constexpr int kWarpsPerBlock = 8;
constexpr int kBlock = kWarpsPerBlock * 32;
constexpr int kSmall = 8;      // largest cluster that a partial table leaves out (see rebuild.cuh)
constexpr int kRunBodies = 512; // sweep bodies of one launch of a run at most, and of the time records
constexpr int kOwnNever = -3;  // own[v].y below every change stamp: A_a is not known

// One contingency entry: the (cluster, label id) key, its count and the
// delta staged by the current sweep.  16 bytes, read as one vector load.
struct __align__(16) Slot {
    unsigned long long key;
    int cnt;
    int dlt;
};

// Static description of a job inside the union.
struct JobInfo {
    long long vo;   // first union vertex
    long long n;    // vertices
    long long go;   // first entry of the job's rows in G and summ
    int k;          // input partitions
    int kp;         // k rounded up to 4
    int lshift;     // s_j
    int narrow;     // 1: every partition has fewer than 2^16 - 1 classes, so G16 holds the labels too
    long long g16;  // first 16-byte word of the job's rows in G16
};

// Per-job state of the current run.
struct JobState {
    unsigned long long nprop;  // |P| of the current sweep
    unsigned long long np1;    // |P1|
    unsigned long long moves;  // moves committed in the current sweep
    long long dF;              // objective change of the current sweep
    long long dF_p1;           // dF of P1 as evaluated
    long long F;               // current objective
    long long recompute;       // F' accumulator (heavy sweeps, recompute)
    long long partition_sq;    // sum_i sum_j |P_ij|^2
    long long t_prop;          // colour_batched: the sweep's totals over its classes so far:
    long long t_p1;            //   |P|, |P1|, dF of P1, classes that fell back, moves
    long long t_dFp1;
    long long t_fb;
    long long t_moves;
    int mode;                  // 0 nothing to commit, 1 commit P1 (staged), 2 matching, 3 P1 committed (rebuilt)
    int stop;                  // 1: this job's run has stopped
    int sweeps;                // sweeps recorded since creation / reset
    int run_sweeps;            // sweeps in the current run
    int rollback;              // 1: this heavy sweep's P1 was rejected and is being undone
    int pad;
};

// Device-resident control block of a context (union-wide state).
struct DevState {
    unsigned long long nprop;    // proposals of the current sweep, all jobs
    unsigned long long pkeys;    // sum over those proposals of their job's k (label rows they move)
    unsigned long long used;     // occupied table slots
    long long live;              // keys with a non-zero count
    unsigned long long mask;     // active table capacity - 1 (a power of two minus one)
    unsigned long long new_mask; // capacity - 1 of a pending rebuild
    int skip;                    // 1: this sweep does nothing (every job has stopped)
    int stop;                    // 1: the run has stopped (all jobs)
    int active;                  // jobs still running after the current sweep
    int rebuild;                 // 1: a table rebuild is pending
    int err;                     // cc_status of a device-side failure (first one wins)
    int overflow;                // 1: the table ran short during this sweep (nothing committed)
    int abort;                   // 1: the pending rebuild follows an abandoned sweep
    int retries;                 // sweeps abandoned and retried in a larger table
    int rebuilds;                // table rebuilds since creation
    int heavy;                   // 1: this sweep evaluates P1 by a rebuild (see sweep.cu)
    int rollback;                // 1: some job's heavy P1 is being undone
    int tvalid;                  // 1: the table holds the counts of the current C
    int run_limit;               // sweep limit of the current run
    int run_until;               // sweep graphs: bodies after which the loop ends
    int run_bodies;              // sweeps of the current run that did work (retried ones included)
    unsigned long long region_launches;  // kernels run inside the gated regions of sweep graphs
    int stamp;                   // number of the current sweep (since creation; retried sweeps reuse it)
    int all_active;              // 1: every vertex is scored in this sweep (first sweep of a run)
    int cls;                     // colour_batched: the class this sweep body runs
    int ncls;                    // colour_batched: number of classes (of the job with the most)
    unsigned long long safe_mask;  // heavy sweep: capacity - 1 that holds every key it can create
    int tight;                   // 1: the pending rebuild tries a capacity below safe_mask (checked)
    int again;                   // 1: the tight attempt was too small; the rebuild runs again at safe_mask
    int build_fail;              // 1: an insert of the tight attempt ran past its probe limit
    int small;                   // clusters of at most this many members have no keys and no summary rows
                                 //    in the table (they are scored from the member list); 0: every
                                 //    cluster has them
    int build_small;             // the same for the pending rebuild
    int build_light;             // heavy sweep: 1 if its proposals would fit a light sweep
    int sized;                   // heavy sweep: the capacity of its rebuild is settled
    unsigned long long small_keys;  // heavy sweep: label rows in clusters of at most kSmall members after P1
    unsigned long long keys_all; // upper estimate of the distinct keys of C at the last rebuild
    unsigned long long retry_mask;  // heavy sweep: capacity - 1 of the second attempt of its rebuild
    int many;                    // 1: many vertices may move (the sweep before moved more than 1/8 of the label rows)
    int match;                   // 1: some job of this sweep falls back to the matching
    long long classes;           // label compaction (in its own control block): classes of all partitions together
    // run kernel (persist.cu); written between two steps only
    int rebuild_kind;            // the running rebuild: 0 heavy sweep, 1 its rollback, 2 end of the sweep
    int tries;                   // rebuild attempts of this heavy sweep
    int bodies_left;             // sweep bodies the launch may still run
    unsigned bar_word;           // barriers passed << 8 | step that follows
    unsigned bar_count;          // blocks that have arrived at the barrier; 0 between launches (left over where
    int bar_abort;               //    a block gave up waiting (1: every block leaves): the host clears both)
};

// Arguments of the kernels (passed by value).
struct SweepArgs {
    long long n;                // N, union vertices
    long long nnz;              // union CSR entries
    int jobs;                   // J
    int kmax;                   // largest k_j
    const long long* off;
    const int* col;
    const int* src;             // source vertex of each CSR entry (nnz)
    const int* jid;             // job of each vertex
    const JobInfo* job;         // J
    JobState* js;               // J
    const int* G;
    const int4* G16;            // label rows again, as 16-bit class numbers (JobInfo::narrow)
    int4* summ;
    int* C;
    int* size;
    int* dsize;                 // staged size deltas
    unsigned long long* best;   // bids: per vertex in the proposal step, per cluster in the matching
    int2* own;                  // per vertex {A_a, change stamp of its cluster when that was computed}
    Slot* table;
    unsigned long long mask_max; // allocated capacity - 1; the active capacity is st->mask + 1
    unsigned long long cap_min;  // smallest active capacity
    unsigned long long keys;     // sum_j k_j n_j: no C has more live keys
    int sweep_mode;              // 0 automatic, 1 always staged deltas, 2 always rebuild
    int gs;                      // lanes that score one item (a power of two, 1..32)
    int gs_set;                  // 1: set by the caller (cc_options.lanes)
    int active_set;              // 1: score only the active vertices (cc_options.active_set)
    int empty_moves;             // 1: a vertex may also move into a new cluster with its own id (cc_options.empty_moves)
    int tight_mode;              // cc_options.tight_rebuild: 0 tight attempt first, 1 never, 2 always dropped
    int colour_mode;             // 1: colour-batched sweeps (cc_options.colour_batched): a sweep body
                                 //    runs the vertices of colour class st->cls only
    const int* vlist;            // colour_batched: vertices listed class by class (n)
    const int* voff;             // colour_batched: first entry of each class in vlist (ncls + 1)
    const int* eidx;             // colour_batched: CSR entries of each class's vertices, class by class (nnz)
    const long long* eoff;       // colour_batched: first entry of each class in eidx (ncls + 1)
    int* chg;                   // per cluster id: stamp of the last sweep that moved a vertex into or out of it
    unsigned long long* prev;   // per vertex: its bid of the last sweep that scored it (kEmpty: none)
    unsigned char* act;         // per vertex: 1 if all its candidates are scored in this sweep
    int* pv;                    // proposal list: vertex,
    int* pa;                    //   source cluster,
    int* pb;                    //   target cluster,
    int* pg;                    //   gain dD
    unsigned char* pflag;       //   1 if kept by the singleton guard (2: matching winner)
    int* members;               // rebuild scratch: vertices listed cluster by cluster (n)
    int* cursor;                // rebuild scratch: next free position of each cluster (n)
    int* bsum;                  // rebuild scratch: per-block sums of the size scan (bsum_entries)
    DevState* st;
    unsigned long long* ts;     // kRunBodies times {start of a sweep body, end of its proposal step, its end} (ns)
    cc_sweep_info* hist;        // J x hist_cap records
    int hist_cap;
    unsigned long long wait_ns; // run kernel: longest wait of a block at a barrier (cc_set_wait_limit)
};

// The block's share of a step's items (each one warp's work, of uneven cost):
// kWarpsPerBlock consecutive ones of every gridDim.x times that many, which
// its warps take one after another from a counter in shared memory, so that
// they end together.  start() is called by the whole block, next() by a whole
// warp; the items are used up when next() passes their number.
struct WarpQueue {
    int* taken;  // shared

    __device__ __forceinline__ void start() const
    {
        __syncthreads();
        if (threadIdx.x == 0) *taken = 0;
        __syncthreads();
    }

    __device__ __forceinline__ long long next() const
    {
        int i = 0;
        if ((threadIdx.x & 31) == 0) i = atomicAdd(taken, 1);
        i = __shfl_sync(0xffffffffu, i, 0);
        return ((long long)(i / kWarpsPerBlock) * gridDim.x + blockIdx.x) * kWarpsPerBlock + i % kWarpsPerBlock;
    }
};

// 16-bit label rows: a job's rows are quads16(k) 16-byte words each, eight
// class numbers to a word.
constexpr int kNoClass16 = 0xffff;  // the padding, and the first number that does not fit

__host__ __device__ __forceinline__ int quads16(int k)
{
    return (k + 7) >> 3;
}

// Row of vertex / cluster x (a union vertex id) of job J in G or summ.
__device__ __forceinline__ long long row_of(const JobInfo& J, long long x)
{
    return J.go + (x - J.vo) * J.kp;
}

// 64-bit finaliser of MurmurHash3 (Austin Appleby, public domain); used by the
// setup-time label map.
__device__ __forceinline__ unsigned long long mix64(unsigned long long z)
{
    z ^= z >> 33;
    z *= 0xff51afd7ed558ccdull;
    z ^= z >> 33;
    z *= 0xc4ceb9fe1a85ec53ull;
    z ^= z >> 33;
    return z;
}

// Slot hash of a (cluster, label id) key: the two 32-bit halves mixed with odd
// multipliers, then the 32-bit MurmurHash3 finaliser.  Capacities stay below
// 2^32 slots.
__device__ __forceinline__ unsigned long long hash_key(unsigned long long key)
{
    unsigned h = ((unsigned)(key >> 32) * 0x9E3779B1u) ^ ((unsigned)key * 0x85EBCA77u);
    h ^= h >> 16;
    h *= 0x85EBCA6Bu;
    h ^= h >> 13;
    h *= 0xC2B2AE35u;
    h ^= h >> 16;
    return h;
}

__device__ __forceinline__ unsigned long long ckey(int c, int g)
{
    return ((unsigned long long)(unsigned)c << 32) | (unsigned)g;
}

// Place of partition i in a summary row: entry b of every quad before entry
// b + 1 of any.  The lanes that score a candidate take consecutive quads and
// read the four entries of theirs one after another, so each of the four loads
// is one run of 16-byte words; with the entries of a quad side by side a load
// touched four times the lines, and sweeps 3 and 4 at k = 50 ran at 90% of the
// L1's throughput (a run at n = 2e6: 22.43 -> 21.42 ms, its heavy evaluations
// 2.96 -> 2.16; n = 1e6, k = 20: 6.50 -> 6.44).
__device__ __forceinline__ int summ_at(const JobInfo& J, int i)
{
    return (i & 3) * (J.kp >> 2) + (i >> 2);
}

// Keeps the summary entry of (cluster x, partition p) of job J exact after the
// count of label g there changed by d: only the counts of the entry's two
// labels are stored.
__device__ __forceinline__ void summ_update(const SweepArgs& a, const JobInfo& J, int x, int p, int g, int d)
{
    int4* S = a.summ + row_of(J, x) + summ_at(J, p);
    const int d1 = S->x, d2 = S->z;
    if (d1 == g) atomicAdd(&S->y, d);
    else if (d2 == g) atomicAdd(&S->w, d);
}

__device__ __forceinline__ void set_err(DevState* st, int code)
{
    atomicCAS(&st->err, 0, code);
}

// Adds x to the 64-bit field of job `job` in an array of JobState (field at
// base, records stride_ll long longs apart): one atomic per warp when all of
// its lanes belong to one job (the usual case), one per lane otherwise.
// Every lane of the warp must call it; job < 0 adds nothing.
__device__ __forceinline__ void job_add64(long long x, int job, long long* base, size_t stride_ll)
{
    const unsigned same = __match_any_sync(0xffffffffu, job);
    if (same == 0xffffffffu) {
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if ((threadIdx.x & 31) == 0 && x != 0 && job >= 0)
            atomicAdd(reinterpret_cast<unsigned long long*>(base + (size_t)job * stride_ll), (unsigned long long)x);
    } else if (x != 0 && job >= 0) {
        atomicAdd(reinterpret_cast<unsigned long long*>(base + (size_t)job * stride_ll), (unsigned long long)x);
    }
}

constexpr size_t kJobStride = sizeof(JobState) / sizeof(long long);

// Per-job 64-bit sums over a kernel's loop: each thread keeps a running
// (job, sum) and flushes it when its job changes -- into a shared-memory
// array of per-job sums when the context has few jobs (sh != nullptr), else
// straight into the job records -- and finish() adds what is left, once per
// warp for one job.  For a single job that is one global atomic per warp per
// launch instead of one per loop iteration.
constexpr int kSmemJobs = 1024;

struct JobAcc {
    int job = -1;
    long long sum = 0;
    long long* sh;      // shared per-job sums or nullptr
    long long* base;    // field of job 0 in the JobState array
    size_t stride;

    __device__ __forceinline__ JobAcc(long long* sh_, long long* base_, size_t stride_)
        : sh(sh_), base(base_), stride(stride_) {}

    __device__ __forceinline__ void flush()
    {
        if (job >= 0 && sum != 0) {
            unsigned long long* dst = reinterpret_cast<unsigned long long*>(sh ? sh + job : base + (size_t)job * stride);
            atomicAdd(dst, (unsigned long long)sum);
        }
        sum = 0;
    }

    __device__ __forceinline__ void add(int j, long long x)
    {
        if (x == 0) return;
        if (j != job) {
            flush();
            job = j;
        }
        sum += x;
    }
};

// Shared per-job sums of a block for contexts of 2..kSmemJobs jobs (dynamic
// shared memory of smem_jobs_bytes(jobs)); nullptr otherwise.  Every thread
// of the block must call it.
__device__ __forceinline__ long long* job_smem_init(int jobs, long long* dyn)
{
    if (jobs < 2 || jobs > kSmemJobs) return nullptr;
    for (int j = threadIdx.x; j < jobs; j += blockDim.x) dyn[j] = 0;
    __syncthreads();
    return dyn;
}

inline size_t smem_jobs_bytes(int jobs)
{
    return (jobs >= 2 && jobs <= kSmemJobs) ? sizeof(long long) * (size_t)jobs : 0;
}

// Adds what the accumulators of the block hold to the job records.  Every
// thread of the block must call it, after its last add().
__device__ __forceinline__ void job_acc_finish(JobAcc& acc, int jobs)
{
    if (acc.sh) {
        acc.flush();
        __syncthreads();
        for (int j = threadIdx.x; j < jobs; j += blockDim.x) {
            const long long x = acc.sh[j];
            if (x != 0) atomicAdd(reinterpret_cast<unsigned long long*>(acc.base + (size_t)j * acc.stride),
                                  (unsigned long long)x);
        }
    } else {
        // lanes that added nothing hold job -1 and sum 0; with one job they
        // join the others so that the warp adds with one atomic
        job_add64(acc.sum, jobs == 1 ? 0 : acc.job, acc.base, acc.stride);
    }
}
static_assert(sizeof(JobState) % sizeof(long long) == 0, "JobState must be a multiple of 8 bytes");

// Slot holding key, or -1 (coherent loads; the key must not be inserted concurrently).
__device__ __forceinline__ long long table_find(const Slot* t, unsigned long long mask, unsigned long long key)
{
    unsigned long long h = hash_key(key) & mask;
    for (unsigned long long p = 0; p <= mask; ++p) {
        unsigned long long k = *reinterpret_cast<const volatile unsigned long long*>(&t[h].key);
        if (k == key) return (long long)h;
        if (k == kEmpty) return -1;
        h = (h + 1) & mask;
    }
    return -1;
}

// Slot holding key, inserting it (count 0, delta 0) if absent.  *inserted is
// set when this call created the slot.  Returns -1 if the table is full.
__device__ __forceinline__ long long table_find_or_insert(Slot* t, unsigned long long mask,
                                                          unsigned long long key, bool* inserted)
{
    *inserted = false;
    unsigned long long h = hash_key(key) & mask;
    for (unsigned long long p = 0; p <= mask; ++p) {
        unsigned long long k = *reinterpret_cast<volatile unsigned long long*>(&t[h].key);
        if (k == key) return (long long)h;
        if (k == kEmpty) {
            unsigned long long old = atomicCAS(&t[h].key, kEmpty, key);
            if (old == kEmpty) { *inserted = true; return (long long)h; }
            if (old == key) return (long long)h;
        }
        h = (h + 1) & mask;
    }
    return -1;
}

// 16-byte compare-and-swap of a summary entry (PTX atom.cas.b128, sm_90 and
// later): returns the entry's previous contents; the swap happened iff they
// equal cmp.
__device__ __forceinline__ ulonglong2 entry_cas(int4* p, ulonglong2 cmp, ulonglong2 val)
{
    ulonglong2 old;
    asm volatile(
        "{\n\t"
        ".reg .b128 c, v, d;\n\t"
        "mov.b128 c, {%2, %3};\n\t"
        "mov.b128 v, {%4, %5};\n\t"
        "atom.relaxed.gpu.global.cas.b128 d, [%6], c, v;\n\t"
        "mov.b128 {%0, %1}, d;\n\t"
        "}"
        : "=l"(old.x), "=l"(old.y)
        : "l"(cmp.x), "l"(cmp.y), "l"(val.x), "l"(val.y), "l"(p)
        : "memory");
    return old;
}

// ---- setup.cu ----
// SMs of the current device (queried once per device; 1 if the query fails).
constexpr int kMaxDevices = 64;
int device_sm_count();

// Union assembly: per-job inputs were copied into staging buffers (offsets of
// job j at offstage[vo_j + j ..], n_j + 1 entries; columns job-local at
// col[eo_j ..]); these kernels validate them, build the union offsets, the
// source array and the job of each vertex, and shift the columns to union ids.
struct AssemblyArgs {
    int jobs;
    long long n, nnz;
    const long long* offstage;  // N + J entries
    const long long* eo;        // J + 1: first CSR entry of each job
    const JobInfo* job;
    long long* off;             // N + 1
    int* col;                   // NNZ, job-local on entry, union ids on exit
    int* src;
    int* jid;
    DevState* st;
};
// (the second does nothing once the first has found the offsets malformed).
cudaError_t launch_assemble(const AssemblyArgs& a, cudaStream_t s);

// Label compaction of all jobs: labels staged partition-major per job (job j's
// k_j x n_j block at lo_j); pjob maps a global partition index (sum of the
// earlier k plus i) to its job, pfirst the job to its first global partition.
struct LabelArgs {
    int jobs;
    const int* labels;          // staged labels
    const long long* lo;        // J + 1: first staged label of each job
    const int* pjob;            // global partition -> job
    const int* pfirst;          // J: first global partition of each job
    JobInfo* job;               // (narrow is cleared where a partition has too many classes)
    JobState* js;
    int* G;
    int4* G16;
    int parts;                  // partitions of all jobs
    int* part_n;                // per global partition: its classes (zeroed)
    void* lmap;                 // 16-byte slots, lmask + 1 of them
    unsigned long long lmask;
    unsigned long long limit;   // probes of an insert before st->err is set to CC_ERR_TABLE_FULL
    unsigned* slots;            // scratch: the map entry of every staged label (total)
    int tiles, turns;           // tiles of the two passes over the labels, and the first of each job
    const int* tile0;
    const int* turn0;
    DevState* st;
    long long* classes;         // label classes of all partitions together
    long long* part_sq;         // per global partition: sum_l |P_il|^2
    double* part_slog;          // per global partition: sum_l |P_il| log |P_il|
};
// Slots of the label map to try first: a quarter of the labels (or 2^16), as
// partitions mostly have few classes for their vertices; `most` holds any.
// An insert that needs more than kLabelProbes probes there gives up
// (st->err = CC_ERR_TABLE_FULL) and the compaction is run again with `most`.
constexpr unsigned long long kLabelProbes = 64;
unsigned long long label_map_slots(long long keys, unsigned long long most);
// Tiles of the passes over the labels, job by job.
struct LabelTiles {
    std::vector<int> tile0, turn0;
    int tiles = 0, turns = 0;
};
void label_tiles(LabelTiles& t, long long n, int k);
// Fills G (padding included), part_sq, part_slog, classes (added to) and the
// jobs' partition_sq (added to).  At most 2^32 map slots.
cudaError_t launch_label_kernels(const LabelArgs& a, cudaStream_t s);

cudaError_t launch_init_state(const SweepArgs& a, int ncls, unsigned long long mask, cudaStream_t s);
// Sizes from C (ids outside their job set CC_ERR_INVALID).
cudaError_t launch_state_from_ids(const SweepArgs& a, cudaStream_t s);
// Rebuild of the table and summary rows from C into st->new_mask + 1 slots,
// then st->mask = st->new_mask.  conditional: only if st->rebuild is set.
// cap: capacity being built, where the host knows it (0: any up to the
// allocated one), for the size of the grids.
cudaError_t launch_table_rebuild(const SweepArgs& a, long long rows, bool conditional, cudaStream_t s,
                                 unsigned long long cap = 0);
// Slots of an empty table.
cudaError_t launch_empty_slots(Slot* t, unsigned long long cap, cudaStream_t s);
// F of every job from scratch into js[j].recompute (without sum_ij |P_ij|^2).
cudaError_t launch_objective_recompute(const SweepArgs& a, cudaStream_t s);

// ---- metrics.cu ----
// Sums for the partition distances of every job's consensus against each of
// its input partitions, from a freshly rebuilt table (its summary rows hold
// each (cluster, partition)'s largest overlap).  Per global partition P (job
// j's partition i is P = pfirst[j] + i): sq[P] = sum n(c,i,l)^2, slog[P] =
// sum n log n, sjc[P] = sum over clusters c of max_l n(c,i,l), sjl[P] = sum
// over classes l of max_c n(c,i,l); per job: csq[j] = sum |c|^2, cslog[j] =
// sum |c| log |c|.  The class maxima are kept in cmap, a hash of the class ids
// with cmask + 1 entries (keys kEmpty, counts 0 at the start), or, where the
// jobs have so many classes that it would be no smaller (cmask 0), in lmax, one
// int per label id of every job (job j's ids start at lbase[j]); all outputs
// zeroed by the caller.
struct MetricsArgs {
    const int* pfirst;
    const long long* lbase;
    long long nlabels;      // entries of lmax
    int* lmax;
    Slot* cmap;
    unsigned long long cmask;
    long long* sq;
    double* slog;
    long long* sjc;
    long long* sjl;
    long long* csq;
    double* cslog;
};
// cap: slots of the table in use.
cudaError_t launch_metrics(const SweepArgs& a, const MetricsArgs& m, int parts, unsigned long long cap, cudaStream_t s);

// Pair (a, b) of input partitions with ka and kb classes: its ka x kb matrix
// starts at cells[off]; its sums.
struct PairDesc {
    int a, b, ka, kb;
    long long off;
};
struct PairSums {
    long long sq;    // sum of n^2 over the cells
    long long rows;  // sum of the row maxima
    long long cols;  // sum of the column maxima
    double slog;     // sum of n log n
};
constexpr int kLogTable = 4096;  // entries of the table of n log n
// ids (k n ints): rank of each vertex's class per partition of job 0,
// partition-major; classes (k ints, zeroed by the caller): classes per
// partition; nlogn: kLogTable doubles.
cudaError_t launch_pair_ids(const SweepArgs& a, int* ids, int* classes, double* nlogn, cudaStream_t s);
// Sums of `count` pairs (at most 65535; cells and out zeroed by the caller;
// kmax: the most classes of a partition).
cudaError_t launch_pairs(long long n, const int* ids, const PairDesc* pairs, int count, int kmax, int* cells,
                         const double* nlogn, PairSums* out, cudaStream_t s);
// C of job j's n vertices := its input partition i (cluster id = least vertex of the class).
cudaError_t launch_ids_from_partition(const SweepArgs& a, long long n, int j, int i, cudaStream_t s);

// Greedy colouring of every job's graph in decreasing splitmix64 priority of
// job-local vertex ids (Jones-Plassmann rounds), then the vertices and CSR
// entries listed class by class; *classes receives the number of classes.
// colour, vlist (n), eidx (nnz), voff / eoff (n + 2 entries) are allocated by
// the caller; cnt (8 (n + 2) bytes) is scratch.
struct ColourArgs {
    long long n, nnz;
    const long long* off;
    const int* col;
    const int* jid;
    const JobInfo* job;
    int* colour;
    int* vlist;
    int* voff;
    int* eidx;
    long long* eoff;
    long long* cnt;
    int* flag;              // one int of scratch
};
cudaError_t launch_colouring(const ColourArgs& a, int* classes, cudaStream_t s);

// ---- api.cu ----
// Message reported by cc_last_error(NULL) in this thread.
void set_thread_error(const std::string& msg);

// ---- sweep.cu ----
// Start of a run of at most `limit` sweeps; a graph's loop ends after `until`
// bodies, which launch_run_more raises to go on with the run.
cudaError_t launch_run_begin(const SweepArgs& a, int limit, int until, cudaStream_t s);
cudaError_t launch_run_more(const SweepArgs& a, int until, cudaStream_t s);
// One sweep of every job.  With a body stream (while s is being captured into a
// graph), the heavy path, its rollback, the light path and the end-of-sweep
// rebuild become IF regions of the graph, each behind a one-thread gate
// kernel, so a sweep launches only the regions it needs.
constexpr int kKernelsPerRebuild = 9;
// regions: heavy path (mark, apply, rebuild), its second rebuild attempt,
// heavy evaluation (eval, decide), rollback (undo, rebuild), light path
// (stage, eval, decide), end-of-sweep rebuild
constexpr int kKernelsInRegions = (2 + kKernelsPerRebuild) + kKernelsPerRebuild + 2 + (1 + kKernelsPerRebuild) + 3 +
                                  kKernelsPerRebuild;
constexpr int kKernelsPerSweep = 11 + kKernelsInRegions;  // kernels of a sweep without regions
constexpr int kGatesPerSweep = 6;
// kernels of a sweep graph outside its regions (gates included); the kernels
// of the regions that run are counted on the device (DevState.region_launches)
constexpr int kKernelsOutsideRegions = kKernelsPerSweep + kGatesPerSweep - kKernelsInRegions;
cudaError_t launch_sweep(const SweepArgs& a, long long rows, int grid, cudaStream_t s, cudaStream_t body);
// Adds to the graph being captured on s a WHILE node whose body (captured on
// `loop`, with the sweep's regions on `body`) is kLoopSweeps sweeps (one after
// the end of the run is skipped) and a gate that repeats them until the run
// stops, fails or has run st->run_until bodies: a whole run as one graph
// launch.
constexpr int kLoopSweeps = 2;
cudaError_t capture_run_loop(const SweepArgs& a, long long rows, int grid, cudaStream_t s, cudaStream_t loop,
                             cudaStream_t body);
cudaError_t prepare_propose(int* blocks_per_sm);
// ---- persist.cu ----
// Blocks of the run kernel: *most are resident at a time on `sms` SMs beside the
// spare places (0: it cannot run), *want is what this context's work fills (one
// thread per CSR entry or vertex and per 8 label rows).
cudaError_t run_grid(const SweepArgs& a, long long rows, int sms, int* most, int* want);
// The run kernel: up to `budget` sweep bodies of a run in one cooperative
// launch (fresh: starts the run first; at most kRunBodies).
cudaError_t launch_run(const SweepArgs& a, long long rows, int grid, int limit, bool fresh, int budget, cudaStream_t s);
// The proposal step's scoring kernels alone (own-cluster sums, candidate
// bids) on the current state, for timing; they write only own, act (the
// same values on the same state) and the bids, which launch_clear_bids
// empties again.  Nothing else of the state changes.
cudaError_t launch_propose_probe(const SweepArgs& a, int grid, cudaStream_t s);
cudaError_t launch_clear_bids(const SweepArgs& a, int grid, cudaStream_t s);

}  // namespace ccg

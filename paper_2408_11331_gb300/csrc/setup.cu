// Setup of the jobs of a context (The algorithm: Initialization) and the
// table maintenance kernels: union assembly with input validation, per-job
// label compaction into the vertex-major membership matrix, the singleton
// state, the contingency hash rebuild with its summary rows, and the
// from-scratch objective used for checks.
#include <algorithm>
#include <atomic>
#include <climits>
#include <vector>

#include "rebuild.cuh"

namespace ccg {

int device_sm_count()
{
    static std::atomic<int> cache[kMaxDevices];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) return 1;
    if (dev < kMaxDevices) {
        const int c = cache[dev].load(std::memory_order_relaxed);
        if (c > 0) return c;
    }
    int sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) return 1;
    if (dev < kMaxDevices) cache[dev].store(sms, std::memory_order_relaxed);
    return sms;
}

namespace {

constexpr int kSetupBlock = 256;

// Grid for grid-stride kernels: one block per kSetupBlock items, at most 16
// resident blocks per SM of the current device.
inline int grid_for(long long work, int per_block = kSetupBlock)
{
    const long long max_blocks = 16LL * device_sm_count();
    long long b = (work + per_block - 1) / per_block;
    if (b < 1) b = 1;
    if (b > max_blocks) b = max_blocks;
    return (int)b;
}

// (global partition, raw label) -> least job-local vertex carrying it, and the class size.
struct __align__(16) LSlot {
    unsigned long long key;
    int rep;
    int cnt;
};

__device__ __forceinline__ int job_of_vertex(const JobInfo* job, int jobs, long long v)
{
    int lo = 0, hi = jobs - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (job[mid].vo <= v) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Largest index i with key[i] <= x among key[0..count) (key[0] <= x assumed).
__device__ __forceinline__ int upper_index32(const int* key, int count, int x)
{
    int lo = 0, hi = count - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (key[mid] <= x) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// ---- union assembly -------------------------------------------------------

// jid[v], and off[v] = eo_j + (job-local offset); checks each job's offsets
// start at 0, do not decrease and end at its nnz.
__global__ void k_assemble_off(AssemblyArgs a)
{
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < a.n; v += stride) {
        const int j = job_of_vertex(a.job, a.jobs, v);
        const JobInfo J = a.job[j];
        const long long vl = v - J.vo;
        const long long* o = a.offstage + J.vo + j;  // the job's n + 1 offsets
        const long long here = o[vl], next = o[vl + 1];
        bool bad = next < here;
        if (vl == 0 && here != 0) bad = true;
        if (vl == J.n - 1 && next != a.eo[j + 1] - a.eo[j]) bad = true;
        if (bad) atomicCAS(&a.st->err, 0, (int)CC_ERR_INVALID);
        a.jid[v] = j;
        a.off[v] = a.eo[j] + here;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) a.off[a.n] = a.nnz;
}

// Source and (union) neighbour of every CSR entry: a warp per 32 vertices, its
// lanes across their entries, each finding its entry's vertex among the 32
// offsets.  Bound by the writes of src (and the reads of col); a thread per
// vertex wrote 32 rows at once, 80 bytes apart (n = 1e6, nnz = 2e7: 192 us for
// sources and columns, now 114).  In dense graphs of few vertices the entries of
// 32 vertices are cut into slices, one warp each (gridDim.y; a clique of 3000:
// creation 2.21 ms with one warp, 0.66 so).  Skipped when the offsets are malformed.
__global__ void k_assemble_edges(AssemblyArgs a)
{
    if (a.st->err) return;
    const int lane = threadIdx.x & 31;
    const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long v0 = (((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 32; v0 < a.n; v0 += nwarps * 32) {
        const long long v = v0 + lane;
        const long long mine = v < a.n ? a.off[v] : a.nnz;
        const long long e0 = __shfl_sync(0xffffffffu, mine, 0);
        const long long e1 = v0 + 32 < a.n ? a.off[v0 + 32] : a.nnz;
        const int at = (int)(mine - e0 < e1 - e0 ? mine - e0 : e1 - e0);  // a row holds fewer than 2^31 entries here
        const bool wide = e1 - e0 >= (1LL << 31);
        const JobInfo J = a.job[a.jid[v < a.n ? v : a.n - 1]];
        for (long long b = e0 + 32 * blockIdx.y; b < e1; b += 32 * gridDim.y) {
            const long long e = b + lane;
            // last of the 32 offsets that is not past e
            int l = 0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const long long x = wide ? __shfl_sync(0xffffffffu, mine, l + o) - e0
                                         : (long long)__shfl_sync(0xffffffffu, at, l + o);
                if (x <= e - e0) l += o;
            }
            const int n = __shfl_sync(0xffffffffu, (int)J.n, l);
            const int vo = __shfl_sync(0xffffffffu, (int)J.vo, l);
            if (e >= e1) continue;
            a.src[e] = (int)(v0 + l);
            const int c = a.col[e];
            if (c < 0 || c >= n) {
                atomicCAS(&a.st->err, 0, (int)CC_ERR_INVALID);
                a.col[e] = vo;
            } else if (vo != 0) {
                a.col[e] = vo + c;
            }
        }
    }
}

// ---- label compaction -----------------------------------------------------

__global__ void k_lmap_clear(LSlot* m, unsigned long long cap)
{
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    for (unsigned long long s = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; s < cap; s += stride)
        reinterpret_cast<ulonglong2*>(m)[s] = make_ulonglong2(kEmpty, (unsigned long long)(unsigned)INT_MAX);
}

// Entry of (global partition, raw label) in the map, inserted if absent, with
// its least vertex lowered to vl; -1 after `limit` probes.  One 16-byte load
// finds the key and tells whether the least vertex is smaller already (it
// mostly is: the vertices come roughly in order).
__device__ __forceinline__ long long lmap_put(LSlot* m, unsigned long long mask, unsigned long long limit,
                                              unsigned long long key, int vl)
{
    unsigned long long h = mix64(key) & mask;
    for (unsigned long long p = 0; p <= mask && p < limit; ++p) {
        const ulonglong2 e = __ldcg(reinterpret_cast<const ulonglong2*>(m + h));
        unsigned long long k = e.x;
        if (k == kEmpty) {
            k = atomicCAS(&m[h].key, kEmpty, key);
            if (k == kEmpty) k = key;
        }
        if (k == key) {
            if ((int)(unsigned)(e.y & 0xffffffffull) > vl || e.x != key) atomicMin(&m[h].rep, vl);
            return (long long)h;
        }
        h = (h + 1) & mask;
    }
    return -1;
}

// Every label of every job: tiles of kTile vertices of one partition.  The
// entry found goes to slots (the next pass then needs no lookup), and the
// class sizes are added once per class and tile: one atomic per label on a
// few thousand words bounded this pass (n = 1e6, k = 20: 1107 us, with the
// 64-bit divisions and job searches per label that the tiles save; now 248).
__global__ void __launch_bounds__(kBlock) k_label_insert(LabelArgs a)
{
    __shared__ TileCount tc;
    LSlot* m = static_cast<LSlot*>(a.lmap);
    for (int tile = blockIdx.x; tile < a.tiles; tile += gridDim.x) {
        // the map has proved too small: the compaction is run again
        if (a.limit != ~0ull && __syncthreads_or(*reinterpret_cast<volatile int*>(&a.st->err))) break;
        const int j = upper_index32(a.tile0, a.jobs, tile);
        const int n = (int)a.job[j].n, per = (n + kTile - 1) / kTile, rel = tile - a.tile0[j];
        const int i = rel / per, v0 = (rel - i * per) * kTile;
        const long long t0 = a.lo[j] + (long long)i * n;
        const unsigned long long part = (unsigned long long)(unsigned)(a.pfirst[j] + i) << 32;
        int id[4], slot[4], rank[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int vl = v0 + q * kBlock + threadIdx.x;
            id[q] = -1;
            if (vl >= n) continue;
            const long long s = lmap_put(m, a.lmask, a.limit, part | (unsigned)a.labels[t0 + vl], vl);
            if (s < 0) {
                set_err(a.st, CC_ERR_TABLE_FULL);
                continue;
            }
            a.slots[t0 + vl] = (unsigned)s;
            if (a.lmask >> 31) atomicAdd(&m[s].cnt, 1);  // (a map too large for the tile's ids)
            else id[q] = (int)s;
        }
        tile_count(&tc, id, slot, rank);
        for (int s = threadIdx.x; s < 2 * kTile; s += kBlock)
            if (tc.cnt[s]) atomicAdd(&m[tc.key[s]].cnt, tc.cnt[s]);
        __syncthreads();
    }
}

// The classes numbered within their partition (the number replaces the raw
// label in the class's key), sum_i sum_j |P_ij|^2 of every job and the sums per
// partition.  With at most kSmemParts partitions a block counts its tile's
// classes and adds up its sums in shared memory, so that a partition's words
// take an add per tile instead of one per class (n = 1e6, k = 20: 96 us; the
// sums alone, with an add per class, took 85).
constexpr int kSmemParts = 512;
__global__ void __launch_bounds__(kBlock) k_label_classes(LabelArgs a, unsigned long long cap)
{
    extern __shared__ long long dyn_jobs[];
    __shared__ int s_n[kSmemParts], s_base[kSmemParts];
    __shared__ unsigned long long s_sq[kSmemParts];
    __shared__ double s_slog[kSmemParts];
    if (a.st->err) return;
    LSlot* m = static_cast<LSlot*>(a.lmap);
    JobAcc acc(job_smem_init(a.jobs, dyn_jobs), &a.js[0].partition_sq, kJobStride);
    const bool shared = a.parts <= kSmemParts;
    if (shared)
        for (int P = threadIdx.x; P < a.parts; P += kBlock) {
            s_sq[P] = 0;
            s_slog[P] = 0;
        }
    int classes = 0;
    for (unsigned long long b0 = (unsigned long long)blockIdx.x * kTile; b0 < cap; b0 += (unsigned long long)gridDim.x * kTile) {
        if (shared)
            for (int P = threadIdx.x; P < a.parts; P += kBlock) s_n[P] = 0;
        __syncthreads();
        int part[4], rank[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const unsigned long long s = b0 + q * kBlock + threadIdx.x;
            part[q] = -1;
            if (s >= cap) continue;
            const ulonglong2 e = reinterpret_cast<const ulonglong2*>(m)[s];
            if (e.x == kEmpty) continue;
            ++classes;
            const int P = part[q] = (int)(e.x >> 32);
            const long long c = (long long)(e.y >> 32);
            acc.add(a.pjob[P], c * c);
            const double cl = (double)c * log((double)c);
            if (shared) {
                rank[q] = atomicAdd(&s_n[P], 1);
                atomicAdd(&s_sq[P], (unsigned long long)(c * c));
                atomicAdd(&s_slog[P], cl);
            } else {
                rank[q] = atomicAdd(&a.part_n[P], 1);
                atomicAdd(reinterpret_cast<unsigned long long*>(a.part_sq + P), (unsigned long long)(c * c));
                atomicAdd(a.part_slog + P, cl);
            }
        }
        if (shared) {
            __syncthreads();
            for (int P = threadIdx.x; P < a.parts; P += kBlock)
                if (s_n[P]) s_base[P] = atomicAdd(&a.part_n[P], s_n[P]);
            __syncthreads();
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int P = part[q];
            if (P < 0) continue;
            const int id = shared ? s_base[P] + rank[q] : rank[q];
            m[b0 + q * kBlock + threadIdx.x].key = ((unsigned long long)(unsigned)P << 32) | (unsigned)id;
            if (id >= kNoClass16) a.job[a.pjob[P]].narrow = 0;
        }
    }
    __syncthreads();
    if (shared)
        for (int P = threadIdx.x; P < a.parts; P += kBlock)
            if (s_sq[P]) {
                atomicAdd(reinterpret_cast<unsigned long long*>(a.part_sq + P), s_sq[P]);
                atomicAdd(a.part_slog + P, s_slog[P]);
            }
    job_acc_finish(acc, a.jobs);
    for (int o = 16; o > 0; o >>= 1) classes += __shfl_xor_sync(0xffffffffu, classes, o);
    if ((threadIdx.x & 31) == 0 && classes)
        atomicAdd(reinterpret_cast<unsigned long long*>(a.classes), (unsigned long long)classes);
}

// G[row(v) + i] = (i << s_j) | rep(i, label), padding entries -1, and the same
// rows as 16-bit class numbers, padding kNoClass16: tiles of 64
// vertices and 32 partitions, turned in shared memory from the partitions'
// order to the vertices' (written straight, each label was a 4-byte store to
// a sector of its own: n = 1e6, k = 20: 719 us, 91 turned, 107 with the
// 16-bit rows).
constexpr int kTurn = 64;
__global__ void __launch_bounds__(kBlock) k_label_assign(LabelArgs a)
{
    if (a.st->err) return;
    __shared__ int turn[kTurn][33];
    __shared__ __align__(4) unsigned short turn16[kTurn][34];
    const ulonglong2* m = static_cast<const ulonglong2*>(a.lmap);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int tile = blockIdx.x; tile < a.turns; tile += gridDim.x) {
        const int j = upper_index32(a.turn0, a.jobs, tile);
        const JobInfo J = a.job[j];
        const int v0 = (tile - a.turn0[j]) * kTurn, words = quads16(J.k) * 4;
        unsigned* const rows16 = reinterpret_cast<unsigned*>(a.G16 + J.g16);
        for (int i0 = 0; i0 < J.kp; i0 += 32) {
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int i = i0 + w * 4 + r;
                const long long t0 = a.lo[j] + (long long)i * J.n + v0;
#pragma unroll
                for (int h = 0; h < kTurn; h += 32) {
                    const int vl = h + lane;
                    int g = -1, id = kNoClass16;
                    if (i < J.k && v0 + vl < J.n) {
                        const ulonglong2 e = m[a.slots[t0 + vl]];
                        g = (i << J.lshift) | (int)(unsigned)(e.y & 0xffffffffull);
                        id = (int)(unsigned)(e.x & 0xffffffffull);
                    }
                    turn[vl][w * 4 + r] = g;
                    turn16[vl][w * 4 + r] = (unsigned short)id;
                }
            }
            __syncthreads();
            for (int vl = w; vl < kTurn; vl += kWarpsPerBlock) {
                if (v0 + vl >= J.n) break;
                if (i0 + lane < J.kp) a.G[J.go + (long long)(v0 + vl) * J.kp + i0 + lane] = turn[vl][lane];
                // two 16-bit entries per lane
                if (lane < 16 && i0 / 2 + lane < words)
                    rows16[(long long)(v0 + vl) * words + i0 / 2 + lane] =
                        *reinterpret_cast<const unsigned*>(&turn16[vl][2 * lane]);
            }
            __syncthreads();
        }
    }
}

// ---- state ----------------------------------------------------------------

// The control block, the job records and the vertices at the singleton start.
// The counters since creation stay (rebuilds, retries, kernels in regions).
__global__ void k_init_state(SweepArgs a, int ncls, unsigned long long mask)
{
    const long long stride = (long long)gridDim.x * blockDim.x;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        DevState s{};
        s.rebuilds = a.st->rebuilds;
        s.retries = a.st->retries;
        s.region_launches = a.st->region_launches;
        s.stop = 1;
        s.ncls = ncls;
        s.mask = s.new_mask = mask;
        *a.st = s;
    }
    for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < a.jobs; j += stride) {
        JobState s{};
        s.partition_sq = a.js[j].partition_sq;
        s.F = s.partition_sq - (long long)a.job[j].k * a.job[j].n;
        s.stop = 1;
        a.js[j] = s;
    }
    for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < a.n; v += stride) {
        a.C[v] = (int)v;
        a.size[v] = 1;
        a.dsize[v] = 0;
        a.best[v] = kEmpty;
        a.chg[v] = -2;  // stamps start at 0: never "the previous sweep"
        a.own[v] = make_int2(0, kOwnNever);
        a.prev[v] = kEmpty;
        a.act[v] = 1;
    }
}

__global__ void k_sizes_zero(SweepArgs a)
{
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < a.n; v += stride) {
        a.size[v] = 0;
        a.dsize[v] = 0;
        a.best[v] = kEmpty;
        a.own[v].y = kOwnNever;
    }
}

// Sizes from a given consensus; an id outside its vertex's job sets an error.
template <int kPer>
__global__ void __launch_bounds__(kBlock) k_count_sizes(SweepArgs a)
{
    constexpr int kThis = kPer * kBlock;
    __shared__ TileCount tc;
    for (long long t0 = (long long)blockIdx.x * kThis; t0 < a.n; t0 += (long long)gridDim.x * kThis) {
        int id[kPer], slot[kPer], rank[kPer];
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            const long long v = t0 + q * kBlock + threadIdx.x;
            id[q] = -1;
            if (v >= a.n) continue;
            const JobInfo& J = a.job[a.jid[v]];
            const long long c = a.C[v];
            if (c < J.vo || c >= J.vo + J.n) set_err(a.st, CC_ERR_INVALID);
            else id[q] = (int)c;
        }
        tile_count(&tc, id, slot, rank);
        for (int s = threadIdx.x; s < 2 * kThis; s += kBlock)
            if (tc.cnt[s]) atomicAdd(&a.size[tc.key[s]], tc.cnt[s]);
        __syncthreads();
    }
}

// ---- table rebuild: the steps of rebuild.cuh as kernels --------------------

// Block sums of size[] over blocks of 1024 entries.
__global__ void __launch_bounds__(1024) k_scan_blocks(SweepArgs a, int conditional)
{
    if (rebuild_off(a.st, conditional)) return;
    __shared__ int wsum[32];
    const long long i = (long long)blockIdx.x * 1024 + threadIdx.x;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int x = i < a.n ? a.size[i] : 0;
    if (to_size(a.st, conditional)) add_small_rows(a.st, i < a.n ? small_rows(a, i, x) : 0);
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if (lane == 0) wsum[w] = x;
    __syncthreads();
    if (w == 0) {
        int y = wsum[lane];
        for (int o = 16; o > 0; o >>= 1) y += __shfl_xor_sync(0xffffffffu, y, o);
        if (lane == 0) a.bsum[blockIdx.x] = y;
    }
}

// Exclusive scan of the nb block sums in place (one block, 1024 threads, each
// owning a contiguous run).
__global__ void __launch_bounds__(1024) k_scan_sums(SweepArgs a, int nb, int conditional)
{
    if (rebuild_off(a.st, conditional)) return;
    __shared__ int wsum[32];
    if (threadIdx.x == 0 && to_size(a.st, conditional)) size_build(a);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int per = (nb + 1023) / 1024;
    const int lo = threadIdx.x * per, hi = min(nb, lo + per);
    int sum = 0;
    for (int b = lo; b < hi; ++b) sum += a.bsum[b];
    int x = warp_incl_scan(sum, lane);
    if (lane == 31) wsum[w] = x;
    __syncthreads();
    if (w == 0) wsum[lane] = warp_incl_scan(wsum[lane], lane);
    __syncthreads();
    int run = x - sum + (w > 0 ? wsum[w - 1] : 0);
    for (int b = lo; b < hi; ++b) {
        const int y = a.bsum[b];
        a.bsum[b] = run;
        run += y;
    }
}

// cursor[c] = exclusive prefix of size[] (the first position of cluster c).
__global__ void __launch_bounds__(1024) k_scan_write(SweepArgs a, int conditional)
{
    if (rebuild_off(a.st, conditional)) return;
    __shared__ int wsum[32];
    const long long i = (long long)blockIdx.x * 1024 + threadIdx.x;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int v = i < a.n ? a.size[i] : 0;
    int x = warp_incl_scan(v, lane);
    if (lane == 31) wsum[w] = x;
    __syncthreads();
    if (w == 0) wsum[lane] = warp_incl_scan(wsum[lane], lane);
    __syncthreads();
    if (i < a.n) a.cursor[i] = a.bsum[blockIdx.x] + x - v + (w > 0 ? wsum[w - 1] : 0);
}

__global__ void k_table_clear(SweepArgs a, long long rows, int conditional)
{
    table_clear_phase(a, rows, conditional);
}

__global__ void k_members_scatter(SweepArgs a, int conditional)
{
    __shared__ TileCount tc;
    members_scatter_phase(a, conditional, &tc);
}

__global__ void __launch_bounds__(kSetupBlock, 6) k_table_build(SweepArgs a, int conditional)
{
    table_build_phase(a, conditional);
}

__global__ void k_summ_top(SweepArgs a, int conditional)
{
    summ_top_phase(a, conditional);
}

__global__ void k_build_check(SweepArgs a, int conditional)
{
    build_check_phase(a, conditional);
}

__global__ void k_table_done(DevState* st, int conditional)
{
    table_done_phase(st, conditional);
}

// Part of the objective of the clusters that a partial table leaves out: their
// sum_keys n^2 is the sum of A_c over their members, counted inside a warp as in
// h_eval_phase (windows overlap, so that each small cluster lies whole in the
// window of its first member).  A full rebuild for the sake of the sum took 165
// of 235 us (n = 1e5, k = 20, after one sweep; 68 so).
__device__ __forceinline__ void objective_small(const SweepArgs& a, int small, JobAcc& acc)
{
    const int step = 32 - small, lane = threadIdx.x & 31;
    const long long stride = (((long long)gridDim.x * blockDim.x) >> 5) * step;
    long long wb = (((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * step;
    for (; wb < a.n; wb += stride) {
        const bool valid = wb + lane < a.n;
        const int v = valid ? a.members[wb + lane] : 0;
        const int c = valid ? a.C[v] : 0, sc = valid ? a.size[c] : 0;
        const long long at = valid ? (long long)a.cursor[c] - sc : 0;  // the cluster's first place in the list
        const bool on = valid && sc <= small && at >= wb && at < wb + step;
        if (!__any_sync(0xffffffffu, on)) continue;
        const unsigned lanes = on ? (~0u >> (32 - sc)) << (int)(at - wb) : 0u;
        const int job = a.jid[v];
        const JobInfo J = a.job[job];
        const int4* row = reinterpret_cast<const int4*>(a.G + row_of(J, v));
        const int k = on ? J.k : 0;
        int sum = 0;
        for (int i = 0; i < a.kmax; i += 4) {
            // (the padding of a row, -1, counts for nothing: i + b < k)
            const int4 g4 = i < k ? __ldg(row + (i >> 2)) : make_int4(-1, -1, -1, -1);
            const int g[4] = {g4.x, g4.y, g4.z, g4.w};
#pragma unroll
            for (int b = 0; b < 4; ++b)
                sum += __popc(__match_any_sync(0xffffffffu, g[b]) & (i + b < k ? lanes : 0u));
        }
        if (on) acc.add(job, -2LL * sum);
    }
}

// F of every job without sum_ij |P_ij|^2: k sum_c s_c^2 - 2 sum_keys n^2.
__global__ void k_objective_recompute(SweepArgs a)
{
    extern __shared__ long long dyn_jobs[];
    JobAcc acc(job_smem_init(a.jobs, dyn_jobs), &a.js[0].recompute, kJobStride);
    const unsigned long long mask = a.st->mask;
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    const unsigned long long t0 = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
    for (unsigned long long t = t0; t < (unsigned long long)a.n; t += stride) {
        const long long s = a.size[t];
        if (s > 0) {
            const int j = a.jid[t];
            acc.add(j, (long long)a.job[j].k * s * s);
        }
    }
    for (unsigned long long t = t0; t <= mask; t += stride) {
        const ulonglong2 e = reinterpret_cast<const ulonglong2*>(a.table)[t];
        const long long c = (int)(unsigned)(e.y & 0xffffffffull);
        if (e.x != kEmpty && c != 0) acc.add(a.jid[(int)(e.x >> 32)], -2 * c * c);
    }
    if (a.st->small > 0) objective_small(a, a.st->small, acc);
    job_acc_finish(acc, a.jobs);
}

__global__ void k_zero_recompute(SweepArgs a)
{
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < a.jobs; j += gridDim.x * blockDim.x)
        a.js[j].recompute = 0;
}

// ---- colouring (colour_batched) ------------------------------------------
// Priority of a job-local vertex id: the first output of splitmix64 (Steele,
// Lea and Flood) seeded with it; a bijection, so priorities are distinct.
__device__ __forceinline__ unsigned long long colour_priority(unsigned long long v)
{
    unsigned long long z = v + 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

__global__ void k_colour_init(ColourArgs a)
{
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < a.n; v += stride) a.colour[v] = -1;
    if (blockIdx.x == 0 && threadIdx.x == 0) *a.flag = 0;
}

// One Jones-Plassmann round: an uncoloured vertex whose higher-priority
// neighbours are all coloured takes the least colour none of them has, which
// is what the greedy colouring in decreasing priority gives it.  A colour, once
// written, is final, so a vertex that sees a neighbour coloured in this same
// round sees its final colour.  *flag counts the vertices left uncoloured.
__global__ void k_colour_round(ColourArgs a)
{
    const long long stride = (long long)gridDim.x * blockDim.x;
    const volatile int* colour = a.colour;
    int left = 0;
    for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < a.n; v += stride) {
        if (colour[v] >= 0) continue;
        const long long vo = a.job[a.jid[v]].vo;
        const unsigned long long pv = colour_priority((unsigned long long)(v - vo));
        const long long e0 = a.off[v], e1 = a.off[v + 1];
        bool ready = true;
        for (long long e = e0; e < e1 && ready; ++e) {
            const int u = a.col[e];
            if (u != v && colour_priority((unsigned long long)(u - vo)) > pv && colour[u] < 0) ready = false;
        }
        if (!ready) {
            ++left;
            continue;
        }
        // least colour not held by a higher-priority neighbour, 64 at a time
        for (int base = 0;; base += 64) {
            unsigned long long used = 0;
            for (long long e = e0; e < e1; ++e) {
                const int u = a.col[e];
                if (u == v || colour_priority((unsigned long long)(u - vo)) <= pv) continue;
                const int cu = colour[u] - base;
                if (cu >= 0 && cu < 64) used |= 1ull << cu;
            }
            if (~used) {
                a.colour[v] = base + __ffsll((long long)~used) - 1;
                break;
            }
        }
    }
    for (int o = 16; o > 0; o >>= 1) left += __shfl_xor_sync(0xffffffffu, left, o);
    if ((threadIdx.x & 31) == 0 && left) atomicAdd(a.flag, left);
}

__global__ void k_colour_max(ColourArgs a)
{
    const long long stride = (long long)gridDim.x * blockDim.x;
    int m = -1;
    for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < a.n; v += stride) m = max(m, a.colour[v]);
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(a.flag, m + 1);
}

// Per class: vertices (cnt[c]) and CSR entries (cnt[classes + 1 + c]).
__global__ void k_colour_count(ColourArgs a, int classes)
{
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < a.n; v += stride) {
        const int c = a.colour[v];
        atomicAdd(reinterpret_cast<unsigned long long*>(a.cnt + c), 1ull);
        atomicAdd(reinterpret_cast<unsigned long long*>(a.cnt + classes + 1 + c),
                  (unsigned long long)(a.off[v + 1] - a.off[v]));
    }
}

// Lists the vertices and the CSR entries of each class (cnt now holds the
// running positions; the order inside a class does not matter).
__global__ void k_colour_place(ColourArgs a, int classes)
{
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < a.n; v += stride) {
        const int c = a.colour[v];
        const long long d = a.off[v + 1] - a.off[v];
        const long long p = (long long)atomicAdd(reinterpret_cast<unsigned long long*>(a.cnt + c), 1ull);
        a.vlist[p] = (int)v;
        const long long q = (long long)atomicAdd(reinterpret_cast<unsigned long long*>(a.cnt + classes + 1 + c),
                                                 (unsigned long long)d);
        for (long long t = 0; t < d; ++t) a.eidx[q + t] = (int)(a.off[v] + t);
    }
}

}  // namespace

cudaError_t launch_colouring(const ColourArgs& a, int* classes, cudaStream_t s)
{
    const int g = grid_for(a.n);
    k_colour_init<<<g, kSetupBlock, 0, s>>>(a);
    cudaError_t e = cudaGetLastError();
    // rounds until every vertex is coloured; each round colours at least the
    // uncoloured vertex of highest priority, so n rounds always suffice
    for (long long round = 0; e == cudaSuccess; ++round) {
        if (round > a.n) return cudaErrorUnknown;
        e = cudaMemsetAsync(a.flag, 0, sizeof(int), s);
        if (e != cudaSuccess) return e;
        k_colour_round<<<g, kSetupBlock, 0, s>>>(a);
        int left = 0;
        e = cudaMemcpyAsync(&left, a.flag, sizeof(int), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) return e;
        if (left == 0) break;
    }
    e = cudaMemsetAsync(a.flag, 0, sizeof(int), s);
    if (e != cudaSuccess) return e;
    k_colour_max<<<g, kSetupBlock, 0, s>>>(a);
    int nc = 0;
    e = cudaMemcpyAsync(&nc, a.flag, sizeof(int), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return e;
    if (nc < 1) nc = 1;
    e = cudaMemsetAsync(a.cnt, 0, sizeof(long long) * 2 * ((size_t)nc + 1), s);
    if (e != cudaSuccess) return e;
    k_colour_count<<<g, kSetupBlock, 0, s>>>(a, nc);
    std::vector<long long> cnt(2 * ((size_t)nc + 1));
    e = cudaMemcpyAsync(cnt.data(), a.cnt, sizeof(long long) * cnt.size(), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return e;
    // class offsets: exclusive prefix sums of the counts
    std::vector<int> voff((size_t)nc + 1, 0);
    std::vector<long long> eoff((size_t)nc + 1, 0), pos(2 * ((size_t)nc + 1), 0);
    for (int c = 0; c < nc; ++c) {
        voff[c + 1] = voff[c] + (int)cnt[c];
        eoff[c + 1] = eoff[c] + cnt[nc + 1 + c];
        pos[c] = voff[c];
        pos[nc + 1 + c] = eoff[c];
    }
    e = cudaMemcpyAsync(a.voff, voff.data(), sizeof(int) * voff.size(), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(a.eoff, eoff.data(), sizeof(long long) * eoff.size(),
                                              cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(a.cnt, pos.data(), sizeof(long long) * pos.size(),
                                              cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return e;
    k_colour_place<<<g, kSetupBlock, 0, s>>>(a, nc);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);  // pos, voff, eoff are host vectors
    *classes = nc;
    return e;
}

cudaError_t launch_assemble(const AssemblyArgs& a, cudaStream_t s)
{
    k_assemble_off<<<grid_for(a.n), kSetupBlock, 0, s>>>(a);
    // slices of about 1024 entries where the vertices leave warps idle
    const long long groups = (a.n + 31) / 32, warps = 16LL * device_sm_count() * kWarpsPerBlock;
    const long long slices = std::max(1LL, std::min(a.nnz / groups / 1024, warps / groups));
    k_assemble_edges<<<dim3((unsigned)grid_for(a.n), (unsigned)slices), kSetupBlock, 0, s>>>(a);
    return cudaGetLastError();
}

unsigned long long label_map_slots(long long keys, unsigned long long most)
{
    unsigned long long c = 1ull << 16;
    while (c < (unsigned long long)keys / 4) c <<= 1;
    return c < most ? c : most;
}

void label_tiles(LabelTiles& t, long long n, int k)
{
    t.tile0.push_back(t.tiles);
    t.turn0.push_back(t.turns);
    t.tiles += k * (int)((n + kTile - 1) / kTile);
    t.turns += (int)((n + kTurn - 1) / kTurn);
}

cudaError_t launch_label_kernels(const LabelArgs& a, cudaStream_t s)
{
    LSlot* m = static_cast<LSlot*>(a.lmap);
    const unsigned long long cap = a.lmask + 1;
    k_lmap_clear<<<grid_for((long long)cap), kSetupBlock, 0, s>>>(m, cap);
    k_label_insert<<<grid_for(a.tiles, 1), kBlock, 0, s>>>(a);
    k_label_classes<<<grid_for((long long)cap, kTile), kBlock, smem_jobs_bytes(a.jobs), s>>>(a, cap);
    k_label_assign<<<grid_for(a.turns, 1), kBlock, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_init_state(const SweepArgs& a, int ncls, unsigned long long mask, cudaStream_t s)
{
    k_init_state<<<grid_for(a.n), kSetupBlock, 0, s>>>(a, ncls, mask);
    return cudaGetLastError();
}

cudaError_t launch_state_from_ids(const SweepArgs& a, cudaStream_t s)
{
    k_sizes_zero<<<grid_for(a.n), kSetupBlock, 0, s>>>(a);
    if (a.n <= kSmallTiles) k_count_sizes<1><<<grid_for(a.n, kBlock), kBlock, 0, s>>>(a);
    else k_count_sizes<4><<<grid_for(a.n, kTile), kBlock, 0, s>>>(a);
    return cudaGetLastError();
}

__global__ void k_empty_slots(Slot* t, unsigned long long cap)
{
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    for (unsigned long long s = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; s < cap; s += stride)
        reinterpret_cast<ulonglong2*>(t)[s] = make_ulonglong2(kEmpty, 0ull);
}

cudaError_t launch_empty_slots(Slot* t, unsigned long long cap, cudaStream_t s)
{
    k_empty_slots<<<grid_for((long long)cap), kSetupBlock, 0, s>>>(t, cap);
    return cudaGetLastError();
}

cudaError_t launch_table_rebuild(const SweepArgs& a, long long rows, bool conditional, cudaStream_t s,
                                 unsigned long long cap)
{
    const long long slots = cap ? (long long)cap : (long long)a.mask_max + 1;
    const int c = conditional ? 1 : 0;
    const int nb = (int)((a.n + 1023) / 1024);
    k_scan_blocks<<<nb, 1024, 0, s>>>(a, c);
    k_scan_sums<<<1, 1024, 0, s>>>(a, nb, c);
    k_scan_write<<<nb, 1024, 0, s>>>(a, c);
    k_table_clear<<<grid_for(std::max(slots, rows)), kSetupBlock, 0, s>>>(a, rows, c);
    k_members_scatter<<<grid_for(a.n, a.n <= kSmallTiles ? kBlock : kTile), kBlock, 0, s>>>(a, c);
    // (a warp per window of 32 members and quad of partitions where the grid has room)
    k_table_build<<<grid_for((a.n + 31) / 32 * ((a.kmax + 3) / 4), kWarpsPerBlock), kSetupBlock, 0, s>>>(a, c);
    k_build_check<<<1, 32, 0, s>>>(a, c);
    k_summ_top<<<grid_for(slots), kSetupBlock, 0, s>>>(a, c);
    k_table_done<<<1, 1, 0, s>>>(a.st, c);
    return cudaGetLastError();
}

cudaError_t launch_objective_recompute(const SweepArgs& a, cudaStream_t s)
{
    k_zero_recompute<<<grid_for(a.jobs), kSetupBlock, 0, s>>>(a);
    const long long work = (long long)a.mask_max + 1 > a.n ? (long long)a.mask_max + 1 : a.n;
    k_objective_recompute<<<grid_for(work), kSetupBlock, smem_jobs_bytes(a.jobs), s>>>(a);
    return cudaGetLastError();
}

}  // namespace ccg

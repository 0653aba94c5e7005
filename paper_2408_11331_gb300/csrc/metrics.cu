// Partition distances between each job's consensus and its input partitions
// (Methods, "Evaluation metrics": Rand / Mirkin distance, split-join
// distance, variation of information), as reductions over the contingency
// table of the consensus.  The host turns the sums into the distances:
//   Mirkin_i  = sum_c |c|^2 + sum_l |P_il|^2 - 2 sum_{c,l} n(c,i,l)^2   (ordered pairs)
//   SJ_i      = 2n - sum_c max_l n(c,i,l) - sum_l max_c n(c,i,l)
//   VI_i      = (sum_c |c| log|c| + sum_l |P_il| log|P_il| - 2 sum n log n) / n
// (the variation of information H(C|P_i) + H(P_i|C) with p = n(c,i,l) / n).
#include <algorithm>
#include <cmath>

#include "cc_internal.cuh"

namespace ccg {

namespace {

constexpr int kMetBlock = 256;

// Grid for grid-stride kernels: at most 8 resident blocks per SM of the current device.
inline int met_grid(long long work)
{
    const long long max_blocks = 8LL * device_sm_count();
    long long b = (work + kMetBlock - 1) / kMetBlock;
    if (b < 1) b = 1;
    if (b > max_blocks) b = max_blocks;
    return (int)b;
}

// Largest index i with key[i] <= x among key[0..count).
__device__ __forceinline__ int job_by_start(const long long* key, int count, long long x)
{
    int lo = 0, hi = count - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (key[mid] <= x) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Per-partition sums go through shared memory when the context has at most
// kSmemParts partitions (one add per block and partition to global memory).
constexpr int kSmemParts = 1024;

// Counts below this many are first counted per partition and value in shared
// memory (most counts are tiny); 0 bins where the partitions leave no room, and
// in tables of up to kPlainSlots slots, where a block has a few hundred slots and
// the bins cost more than their adds (n = 1000, k = 10: 11.8 us, 9.7 without).
constexpr int kCountBins = 64;
constexpr unsigned long long kPlainSlots = 1ull << 16;

inline int count_bins(int parts, unsigned long long cap)
{
    const int bins = parts <= kSmemParts && cap > kPlainSlots ? 8192 / parts : 0;
    return bins > kCountBins ? kCountBins : bins;
}

// Entry of a label class in the map of class maxima (see MetricsArgs).
__device__ __forceinline__ void class_max(const MetricsArgs& m, unsigned long long id, int cnt)
{
    if (!m.cmask) {
        atomicMax(m.lmax + id, cnt);
        return;
    }
    unsigned long long h = (id * 0x9E3779B97F4A7C15ull >> 24) & m.cmask;
    for (unsigned long long p = 0; p <= m.cmask; ++p) {
        unsigned long long* k = &m.cmap[h].key;
        unsigned long long old = *reinterpret_cast<volatile unsigned long long*>(k);
        if (old == kEmpty) old = atomicCAS(k, kEmpty, id);
        if (old == kEmpty || old == id) {
            atomicMax(&m.cmap[h].cnt, cnt);
            return;
        }
        h = (h + 1) & m.cmask;
    }
}

// Table slots: sum n^2 and sum n log n per partition, max over clusters per
// label.  Bound by the scan of the table; the sums were bound by atomics on
// one word per partition (the slots of a warp hold a few dozen partitions,
// and a shared double add is a compare-and-swap loop: 0.5 ms for 1e6 keys of
// 24 partitions), so counts below `bins` are tallied as integers and turned
// into the sums once per block.
__global__ void k_met_table(SweepArgs a, MetricsArgs m, int parts, int bins)
{
    extern __shared__ unsigned char smem[];
    const bool shared = parts <= kSmemParts;
    long long* ssq = reinterpret_cast<long long*>(smem);
    double* sslog = reinterpret_cast<double*>(smem + sizeof(long long) * (shared ? parts : 0));
    int* tally = reinterpret_cast<int*>(smem + 2 * sizeof(long long) * (shared ? parts : 0));
    if (shared) {
        for (int P = threadIdx.x; P < parts; P += blockDim.x) {
            ssq[P] = 0;
            sslog[P] = 0.0;
        }
        for (int t = threadIdx.x; t < parts * bins; t += blockDim.x) tally[t] = 0;
        __syncthreads();
    }
    long long* sq = shared ? ssq : m.sq;
    double* slog = shared ? sslog : m.slog;
    const unsigned long long cap = a.st->mask + 1;
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    for (unsigned long long s = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; s < cap; s += stride) {
        const ulonglong2 e = reinterpret_cast<const ulonglong2*>(a.table)[s];
        const int cnt = (int)(unsigned)(e.y & 0xffffffffull);
        if (e.x == kEmpty || cnt <= 0) continue;
        const int x = (int)(e.x >> 32), g = (int)(unsigned)(e.x & 0xffffffffull);
        const int j = a.jid[x];
        const int P = m.pfirst[j] + (g >> a.job[j].lshift);
        const long long c = cnt;
        if (cnt < bins) {
            atomicAdd(&tally[P * bins + cnt], 1);
        } else {
            atomicAdd(reinterpret_cast<unsigned long long*>(sq + P), (unsigned long long)(c * c));
            atomicAdd(slog + P, (double)c * log((double)c));
        }
        class_max(m, (unsigned long long)(m.lbase[j] + g), cnt);
    }
    if (shared) {
        __syncthreads();
        for (int t = threadIdx.x; t < parts * bins; t += blockDim.x) {
            const long long many = tally[t], c = t % bins;
            if (many == 0) continue;
            atomicAdd(reinterpret_cast<unsigned long long*>(ssq + t / bins), (unsigned long long)(many * c * c));
            if (c > 1) atomicAdd(sslog + t / bins, (double)many * ((double)c * log((double)c)));
        }
        __syncthreads();
        for (int P = threadIdx.x; P < parts; P += blockDim.x) {
            if (ssq[P]) atomicAdd(reinterpret_cast<unsigned long long*>(m.sq + P), (unsigned long long)ssq[P]);
            if (sslog[P] != 0.0) atomicAdd(m.slog + P, sslog[P]);
        }
    }
}

// Clusters: |c|^2 and |c| log |c| per job, and the largest overlap of each
// (cluster, partition) -- the count of the summary row's label, exact after
// a rebuild.
__global__ void k_met_clusters(SweepArgs a, MetricsArgs m, int parts)
{
    extern __shared__ unsigned char smem[];
    const bool shared = parts <= kSmemParts;
    long long* ssjc = reinterpret_cast<long long*>(smem);
    if (shared) {
        for (int P = threadIdx.x; P < parts; P += blockDim.x) ssjc[P] = 0;
        __syncthreads();
    }
    long long* sjc = shared ? ssjc : m.sjc;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long x = (long long)blockIdx.x * blockDim.x + threadIdx.x; x < a.n; x += stride) {
        const long long s = a.size[x];
        if (s <= 0) continue;
        const int j = a.jid[x];
        const JobInfo& J = a.job[j];
        atomicAdd(reinterpret_cast<unsigned long long*>(m.csq + j), (unsigned long long)(s * s));
        atomicAdd(m.cslog + j, (double)s * log((double)s));
        const int4* S = a.summ + row_of(J, x);
        const int P0 = m.pfirst[j];
        for (int i = 0; i < J.k; ++i)
            atomicAdd(reinterpret_cast<unsigned long long*>(sjc + P0 + i), (unsigned long long)S[summ_at(J, i)].y);
    }
    if (shared) {
        __syncthreads();
        for (int P = threadIdx.x; P < parts; P += blockDim.x)
            if (ssjc[P]) atomicAdd(reinterpret_cast<unsigned long long*>(m.sjc + P), (unsigned long long)ssjc[P]);
    }
}

// Label classes: the largest overlap of each class with a cluster.
__global__ void k_met_labels(SweepArgs a, MetricsArgs m)
{
    const long long stride = (long long)gridDim.x * blockDim.x;
    const long long total = m.cmask ? (long long)m.cmask + 1 : m.nlabels;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += stride) {
        long long id = t;
        int best = 0;
        if (m.cmask) {
            const unsigned long long k = m.cmap[t].key;
            if (k == kEmpty) continue;
            id = (long long)k;
            best = m.cmap[t].cnt;
        } else {
            best = m.lmax[t];
        }
        if (best <= 0) continue;
        const int j = job_by_start(m.lbase, a.jobs, id);
        const int P = m.pfirst[j] + (int)((id - m.lbase[j]) >> a.job[j].lshift);
        atomicAdd(reinterpret_cast<unsigned long long*>(m.sjl + P), (unsigned long long)best);
    }
}

// ---- distances between the input partitions of one job ----------------------
// The k (k - 1) / 2 pairs of partitions as dense contingency matrices: label
// ids are ranked per partition (any order: only equality counts), a cell per
// pair of classes is counted with one atomic per vertex, and the sums and
// maxima are read off the matrix.  Per partition as a consensus, with a
// contingency hash, its summary rows and a reduction (about 0.8 ms each at
// n = 2e5), all 24 x 24 took 25.1 ms; this takes 1.5 ms, most of it the
// counting (55M atomics, 0.53 ms) and the allocations.

// ids[i n + r] = rank of the class of partition i whose least vertex is r.
__global__ void k_pair_ids(SweepArgs a, int* ids, int* classes)
{
    const JobInfo J = a.job[0];
    const int mask = (1 << J.lshift) - 1;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < J.n; v += stride) {
        const int4* row = reinterpret_cast<const int4*>(a.G + v * J.kp);
        for (int q = 0; q < J.kp >> 2; ++q) {
            const int4 g4 = __ldg(row + q);
            const int g[4] = {g4.x, g4.y, g4.z, g4.w};
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const int i = 4 * q + b;
                if (i < J.k && (g[b] & mask) == (int)v) ids[(long long)i * J.n + v] = atomicAdd(&classes[i], 1);
            }
        }
    }
}

// ids[i n + v] = the rank of v's class, for every other vertex (in place: the
// entries read are those of the least vertices, which keep theirs).
__global__ void k_pair_fill(SweepArgs a, int* ids)
{
    const JobInfo J = a.job[0];
    const int mask = (1 << J.lshift) - 1;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < J.n; v += stride) {
        const int4* row = reinterpret_cast<const int4*>(a.G + v * J.kp);
        for (int q = 0; q < J.kp >> 2; ++q) {
            const int4 g4 = __ldg(row + q);
            const int g[4] = {g4.x, g4.y, g4.z, g4.w};
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const int i = 4 * q + b, r = g[b] & mask;
                if (i < J.k && r != (int)v) ids[(long long)i * J.n + v] = ids[(long long)i * J.n + r];
            }
        }
    }
}

// One atomic per vertex and pair; both id arrays are read in order.
__global__ void k_pair_count(long long n, const int* __restrict__ ids, const PairDesc* __restrict__ pairs, int* cells)
{
    const PairDesc p = pairs[blockIdx.y];
    const int* A = ids + (long long)p.a * n;
    const int* B = ids + (long long)p.b * n;
    int* M = cells + p.off;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride)
        atomicAdd(&M[(long long)A[v] * p.kb + B[v]], 1);
}

__global__ void k_nlogn(double* t)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c < kLogTable) t[c] = c > 1 ? (double)c * log((double)c) : 0.0;
}

// A warp per row of the matrix: sum n^2, sum n log n, the row maxima's sum.
__global__ void __launch_bounds__(kMetBlock) k_pair_rows(const PairDesc* __restrict__ pairs, const int* __restrict__ cells,
                                                         const double* __restrict__ nlogn, PairSums* out)
{
    __shared__ long long s_sq, s_max;
    __shared__ double s_log;
    if (threadIdx.x == 0) {
        s_sq = s_max = 0;
        s_log = 0.0;
    }
    __syncthreads();
    const PairDesc p = pairs[blockIdx.y];
    const int lane = threadIdx.x & 31, warps = kMetBlock / 32;
    long long sq = 0, mx = 0;
    double lg = 0.0;
    for (int r = blockIdx.x * warps + (threadIdx.x >> 5); r < p.ka; r += gridDim.x * warps) {
        const int* row = cells + p.off + (long long)r * p.kb;
        int top = 0;
        for (int c = lane; c < p.kb; c += 32) {
            const int x = row[c];
            if (x == 0) continue;
            top = max(top, x);
            sq += (long long)x * x;
            lg += x < kLogTable ? nlogn[x] : (double)x * log((double)x);
        }
        top = __reduce_max_sync(0xffffffffu, top);
        if (lane == 0) mx += top;
    }
    for (int o = 16; o > 0; o >>= 1) {
        sq += __shfl_xor_sync(0xffffffffu, sq, o);
        lg += __shfl_xor_sync(0xffffffffu, lg, o);
    }
    if (lane == 0) {
        atomicAdd(reinterpret_cast<unsigned long long*>(&s_sq), (unsigned long long)sq);
        atomicAdd(reinterpret_cast<unsigned long long*>(&s_max), (unsigned long long)mx);
        atomicAdd(&s_log, lg);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        PairSums* o = out + blockIdx.y;
        if (s_sq) atomicAdd(reinterpret_cast<unsigned long long*>(&o->sq), (unsigned long long)s_sq);
        if (s_max) atomicAdd(reinterpret_cast<unsigned long long*>(&o->rows), (unsigned long long)s_max);
        if (s_log != 0.0) atomicAdd(&o->slog, s_log);
    }
}

// A thread per column: the column maxima's sum.
__global__ void __launch_bounds__(kMetBlock) k_pair_cols(const PairDesc* __restrict__ pairs, const int* __restrict__ cells,
                                                         PairSums* out)
{
    const PairDesc p = pairs[blockIdx.y];
    long long mx = 0;
    for (int c = blockIdx.x * kMetBlock + threadIdx.x; c < p.kb; c += gridDim.x * kMetBlock) {
        const int* col = cells + p.off + c;
        int top = 0;
        int r = 0;
        for (; r + 8 <= p.ka; r += 8) {
            int x[8];
#pragma unroll
            for (int b = 0; b < 8; ++b) x[b] = col[(long long)(r + b) * p.kb];
#pragma unroll
            for (int b = 0; b < 8; ++b) top = max(top, x[b]);
        }
        for (; r < p.ka; ++r) top = max(top, col[(long long)r * p.kb]);
        mx += top;
    }
    for (int o = 16; o > 0; o >>= 1) mx += __shfl_xor_sync(0xffffffffu, mx, o);
    if ((threadIdx.x & 31) == 0 && mx) atomicAdd(reinterpret_cast<unsigned long long*>(&out[blockIdx.y].cols),
                                                (unsigned long long)mx);
}

// C := input partition i of job j as a consensus: every vertex in the cluster
// named by the least vertex of its class (the representative in its label id).
__global__ void k_ids_from_partition(SweepArgs a, int j, int i)
{
    const JobInfo J = a.job[j];
    const int mask = (1 << J.lshift) - 1;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long v = J.vo + (long long)blockIdx.x * blockDim.x + threadIdx.x; v < J.vo + J.n; v += stride)
        a.C[v] = (int)(J.vo + (a.G[row_of(J, v) + i] & mask));
}

}  // namespace

cudaError_t launch_ids_from_partition(const SweepArgs& a, long long n, int j, int i, cudaStream_t s)
{
    k_ids_from_partition<<<met_grid(n), kMetBlock, 0, s>>>(a, j, i);
    return cudaGetLastError();
}

cudaError_t launch_metrics(const SweepArgs& a, const MetricsArgs& m, int parts, unsigned long long cap, cudaStream_t s)
{
    const int bins = count_bins(parts, cap);
    const size_t sm = parts <= kSmemParts ? (size_t)parts * (16 + 4 * (size_t)bins) : 0;
    const size_t sm1 = parts <= kSmemParts ? (size_t)parts * 8 : 0;
    k_met_table<<<met_grid((long long)cap), kMetBlock, sm, s>>>(a, m, parts, bins);
    k_met_clusters<<<met_grid(a.n), kMetBlock, sm1, s>>>(a, m, parts);
    k_met_labels<<<met_grid(m.cmask ? (long long)m.cmask + 1 : m.nlabels), kMetBlock, 0, s>>>(a, m);
    return cudaGetLastError();
}

cudaError_t launch_pair_ids(const SweepArgs& a, int* ids, int* classes, double* nlogn, cudaStream_t s)
{
    k_pair_ids<<<met_grid(a.n), kMetBlock, 0, s>>>(a, ids, classes);
    k_pair_fill<<<met_grid(a.n), kMetBlock, 0, s>>>(a, ids);
    k_nlogn<<<kLogTable / 128, 128, 0, s>>>(nlogn);
    return cudaGetLastError();
}

cudaError_t launch_pairs(long long n, const int* ids, const PairDesc* pairs, int count, int kmax, int* cells,
                         const double* nlogn, PairSums* out, cudaStream_t s)
{
    const int warps = kMetBlock / 32;
    const unsigned gc = (unsigned)std::min<long long>((n + 8 * kMetBlock - 1) / (8 * kMetBlock), 1024);
    const unsigned gr = (unsigned)std::min((kmax + 4 * warps - 1) / (4 * warps), 64);
    const unsigned gl = (unsigned)std::min((kmax + kMetBlock - 1) / kMetBlock, 64);
    k_pair_count<<<dim3(gc, (unsigned)count), kMetBlock, 0, s>>>(n, ids, pairs, cells);
    k_pair_rows<<<dim3(gr, (unsigned)count), kMetBlock, 0, s>>>(pairs, cells, nlogn, out);
    k_pair_cols<<<dim3(gl, (unsigned)count), kMetBlock, 0, s>>>(pairs, cells, out);
    return cudaGetLastError();
}

}  // namespace ccg

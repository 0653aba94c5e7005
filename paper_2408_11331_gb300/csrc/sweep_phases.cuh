// Device code of the sweep's steps (see sweep.cu for the method and for the
// kernels that run one step each, persist.cu for the run kernel that calls
// them between its grid barriers).  Every function is one step over the whole
// grid: blocks take their share by blockIdx and gridDim.
#pragma once

#include "context.cuh"

namespace ccg {

namespace {

constexpr unsigned kFull = 0xffffffffu;

// The device's clock (ns), for the time records of a run.
__device__ __forceinline__ unsigned long long now_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

// (dD, id) packed so that unsigned order is (dD, id) order: dD with its sign
// bit flipped in the high word.
__device__ __forceinline__ unsigned long long pack_key(int dD, int id)
{
    return ((unsigned long long)((unsigned)dD ^ 0x80000000u) << 32) | (unsigned)id;
}

__device__ __forceinline__ int key_gain(unsigned long long key)
{
    return (int)((unsigned)(key >> 32) ^ 0x80000000u);
}

__device__ __forceinline__ long long warp_sum64(long long x)
{
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
    return x;
}

// Adds the warp's sum of x to *out (one atomic).  All lanes must call it.
__device__ __forceinline__ void warp_add64(long long x, long long* out)
{
    x = warp_sum64(x);
    if ((threadIdx.x & 31) == 0 && x != 0) atomicAdd(reinterpret_cast<unsigned long long*>(out), (unsigned long long)x);
}

// Count under key given the slot h = hash(key) & mask already loaded as e.
__device__ __forceinline__ int resolve(const Slot* t, unsigned long long mask, unsigned long long key,
                                       unsigned long long h, ulonglong2 e)
{
    for (unsigned long long p = 0; p <= mask; ++p) {
        if (e.x == key) return (int)(unsigned)(e.y & 0xffffffffull);
        if (e.x == kEmpty) return 0;
        h = (h + 1) & mask;
        e = *reinterpret_cast<const ulonglong2*>(t + h);
    }
    return 0;
}

__device__ __forceinline__ void run_begin_phase(const SweepArgs& a, int limit, int until, int t0, int stride)
{
    DevState* st = a.st;
    if (t0 == 0) {
        st->stop = 0;
        st->run_limit = limit;
        st->run_until = until;
        st->run_bodies = 0;
        st->all_active = 1;
        st->cls = 0;
    }
    for (int j = t0; j < a.jobs; j += stride) {
        a.js[j].stop = 0;
        a.js[j].run_sweeps = 0;
    }
}

__device__ __forceinline__ void begin_phase(const SweepArgs& a, int t0, int stride)
{
    DevState* st = a.st;
    if (t0 == 0) {
        st->skip = (st->stop || st->err) ? 1 : 0;
        if (!st->skip) st->stamp += 1;
        st->many = st->all_active || st->pkeys * 8 > a.keys;
        st->nprop = 0;
        st->pkeys = 0;
        st->overflow = 0;
        st->heavy = 0;
        st->rollback = 0;
        st->active = 0;
        st->tight = 0;
        st->again = 0;
        st->build_fail = 0;
        st->match = 0;
    }
    for (int j = t0; j < a.jobs; j += stride) {
        JobState& s = a.js[j];
        s.nprop = 0;
        s.np1 = 0;
        s.moves = 0;
        s.dF = 0;
        s.dF_p1 = 0;
        s.mode = 0;
        s.rollback = 0;
        s.recompute = 0;
    }
}

constexpr int kInflight = 4;  // loads per lane issued before the first is used

// Job 0, whose vertices and rows start at 0 (the only job with kSingle; the
// known zeros spare address arithmetic and registers).
__device__ __forceinline__ JobInfo first_job(const SweepArgs& a)
{
    JobInfo J;
    J.vo = 0;
    J.go = 0;
    J.n = a.job[0].n;
    J.k = a.job[0].k;
    J.kp = a.job[0].kp;
    J.lshift = 0;
    J.narrow = a.job[0].narrow;
    J.g16 = 0;
    return J;
}

__device__ __forceinline__ int group_sum(int x, int gs)
{
    for (int o = gs >> 1; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
    return x;
}

// The partitions of a job are scored four at a time ("quads"): partition
// 4q + t is component t of quad q of v's label row (one int4 load) and entry
// q + t kp / 4 of x's summary row (one int4 {d1, m1, d2, m2} per partition).  Rows
// are kp = k rounded up to 4 entries; the padding (label -1, summary {-1, 0,
// -1, 0}) adds nothing to the sums below and is never probed.  Lane l of a
// group takes quads l, l + gs, ...  (One partition per lane, with contiguous
// 16-byte entries across a group, measured 10% slower: the scoring is bound
// by instructions, not by L1 lookups.)

// Adds one partition to the summary sums: v's label g against the entry e =
// {d1, m1, d2, m2} of a cluster of size sx.  A label other than d1, d2 has at
// most sx - m1 - m2 members (none when the two cover the cluster).
__device__ __forceinline__ void summary_one(int g, int4 e, int sx, int& ex, int& open)
{
    const bool c1 = g == e.x, c2 = g == e.z;
    ex += c1 ? e.y : (c2 ? e.w : 0);
    if (!(c1 || c2)) open += sx - e.y - e.w;
}

// Summary part of A_x(v) for a non-singleton cluster x (size sx) of job J:
// ex = the counts of v's labels where they are one of the row's two labels
// (exact there; 0, also exact, where the two cover the cluster), ub = ex +
// sum of (sx - m1 - m2) over the other partitions, an upper bound on A_x.
__device__ __forceinline__ void summary_part(const SweepArgs& a, const JobInfo& J, const int* __restrict__ gv, int x,
                                             int sx, int l, int gs, int& ex, int& ub)
{
    ex = 0;
    int open = 0;
    const int4* G4 = reinterpret_cast<const int4*>(gv);
    const int4* S4 = a.summ + row_of(J, x);
    const int kq = J.kp >> 2;
    for (int q = l; q < kq; q += gs) {
        const int4 g = __ldg(G4 + q);
        const int4 e0 = S4[q], e1 = S4[q + kq], e2 = S4[q + 2 * kq], e3 = S4[q + 3 * kq];
        summary_one(g.x, e0, sx, ex, open);
        summary_one(g.y, e1, sx, ex, open);
        summary_one(g.z, e2, sx, ex, open);
        summary_one(g.w, e3, sx, ex, open);
    }
    ub = ex + open;
}

// Starts the probe of one partition if the summary leaves it open (v carries
// neither of the row's labels and the two do not cover x): the contents of
// the key's first slot.
__device__ __forceinline__ bool probe_start(const Slot* __restrict__ table, unsigned long long mask, int x, int g,
                                            int4 e, int sx, ulonglong2& ev)
{
    if (g == e.x || g == e.z || sx <= e.y + e.w) return false;
    ev = *reinterpret_cast<const ulonglong2*>(table + (hash_key(ckey(x, g)) & mask));
    return true;
}

// Exact counts of the partitions the summary leaves open, by hash probes
// (four in flight per lane; key and slot are computed again after the load,
// so only the loaded slots are live while they are in flight).
__device__ __forceinline__ int probe_part(const SweepArgs& a, const JobInfo& J, const Slot* __restrict__ table,
                                          unsigned long long mask, const int* __restrict__ gv, int x, int sx, int l,
                                          int gs)
{
    const int4* G4 = reinterpret_cast<const int4*>(gv);
    const int4* S4 = a.summ + row_of(J, x);
    const int kq = J.kp >> 2;
    int acc = 0;
    for (int q = l; q < kq; q += gs) {
        const int4 g = __ldg(G4 + q);
        ulonglong2 ev[4];
        bool on[4];
        on[0] = probe_start(table, mask, x, g.x, S4[q], sx, ev[0]);
        on[1] = probe_start(table, mask, x, g.y, S4[q + kq], sx, ev[1]);
        on[2] = probe_start(table, mask, x, g.z, S4[q + 2 * kq], sx, ev[2]);
        on[3] = probe_start(table, mask, x, g.w, S4[q + 3 * kq], sx, ev[3]);
        const int gq[4] = {g.x, g.y, g.z, g.w};
#pragma unroll
        for (int b = 0; b < 4; ++b)
            if (on[b]) {
                const unsigned long long key = ckey(x, gq[b]);
                acc += resolve(table, mask, key, hash_key(key) & mask, ev[b]);
            }
    }
    return acc;
}

__device__ __forceinline__ int quad_matches(int4 r, int4 s)
{
    return (r.x == s.x) + (r.y == s.y) + (r.z == s.z) + (r.w == s.w);
}

// This lane's share of A_x(v) for a small cluster, exact: v's label row
// compared with the rows of the members, which the last rebuild listed at
// members[cursor[x] - sx ...) (two of them in flight).  A row is 4 kp bytes,
// a summary row 16 kp, so up to about four members this also reads less.
__device__ __forceinline__ int member_part(const SweepArgs& a, const JobInfo& J, const int* __restrict__ gv, int x,
                                           int sx, int l, int gs)
{
    const int4* G4 = reinterpret_cast<const int4*>(gv);
    const int kq = J.kp >> 2;
    const int* mem = a.members + (a.cursor[x] - sx);
    int acc = l == 0 ? -sx * (J.kp - J.k) : 0;  // the padding matches in every row
    for (int q = l; q < kq; q += gs) {
        const int4 g = __ldg(G4 + q);
        for (int m = 0; m < sx; m += 2) {
            const bool two = m + 1 < sx;
            const int u0 = mem[m], u1 = two ? mem[m + 1] : u0;
            const int4 r0 = __ldg(reinterpret_cast<const int4*>(a.G + row_of(J, u0)) + q);
            const int4 r1 = __ldg(reinterpret_cast<const int4*>(a.G + row_of(J, u1)) + q);
            acc += quad_matches(r0, g);
            if (two) acc += quad_matches(r1, g);
        }
    }
    return acc;
}

// Partitions in which u and v carry the same label, plus the padding entries
// of this lane's quads: the two label rows (kq quads each) compared as int4.
// u's row is a random gather, so its loads go out first; v's row is shared by
// the other candidates of v and mostly in L1.
__device__ __forceinline__ int row_part(const int* gu_row, const int* gv_row, int kq, int l, int gs)
{
    const int4* gu = reinterpret_cast<const int4*>(gu_row);
    const int4* gw = reinterpret_cast<const int4*>(gv_row);
    int acc = 0;
    for (int q0 = l; q0 < kq; q0 += gs * kInflight) {
        int4 r[kInflight];
#pragma unroll
        for (int b = 0; b < kInflight; ++b) {
            const int q = q0 + b * gs;
            r[b] = make_int4(-3, -3, -3, -3);
            if (q < kq) r[b] = __ldg(gu + q);
        }
#pragma unroll
        for (int b = 0; b < kInflight; ++b) {
            const int q = q0 + b * gs;
            if (q < kq) acc += quad_matches(r[b], __ldg(gw + q));
        }
    }
    return acc;  // includes the kp - k padding entries (-1 in every row)
}

// Equal halves among the four words of r and s: a half of x = r ^ s is zero
// where adding 0x7fff to its low 15 bits leaves bit 15 of the sum and of x
// clear.  The words' bits are shifted apart and counted together.
__device__ __forceinline__ unsigned halves_differ(int r, int s)
{
    const unsigned x = (unsigned)(r ^ s);
    return (((x & 0x7fff7fffu) + 0x7fff7fffu) | x) & 0x80008000u;
}

__device__ __forceinline__ int octet_matches(int4 r, int4 s)
{
    return 8 - __popc(halves_differ(r.x, s.x) | (halves_differ(r.y, s.y) >> 1) | (halves_differ(r.z, s.z) >> 2) |
                      (halves_differ(r.w, s.w) >> 3));
}

// This lane's share of the number of partitions in which vertices u and v of
// job J carry the same label.  Where the classes fit 16 bits the rows are half
// as long: the compares of the first sweeps wait for gathered rows (a run at
// n = 2e6, k = 50: 25.38 -> 22.54 ms; n = 1e6, k = 20: 6.85 -> 6.58).
__device__ __forceinline__ int same_part(const SweepArgs& a, const JobInfo& J, long long u, long long v, int l, int gs)
{
    if (!J.narrow) {
        const int part = row_part(a.G + row_of(J, u), a.G + row_of(J, v), J.kp >> 2, l, gs);
        return l == 0 ? part - (J.kp - J.k) : part;
    }
    const int kq = quads16(J.k);
    const int4* gu = a.G16 + (J.g16 + (u - J.vo) * kq);
    const int4* gw = a.G16 + (J.g16 + (v - J.vo) * kq);
    int acc = l == 0 ? J.k - 8 * kq : 0;  // the padding matches
    for (int q0 = l; q0 < kq; q0 += gs * kInflight) {
        int4 r[kInflight];
#pragma unroll
        for (int b = 0; b < kInflight; ++b) {
            const int q = q0 + b * gs;
            r[b] = make_int4(0, 0, 0, 0);
            if (q < kq) r[b] = __ldg(gu + q);
        }
#pragma unroll
        for (int b = 0; b < kInflight; ++b) {
            const int q = q0 + b * gs;
            if (q < kq) acc += octet_matches(r[b], __ldg(gw + q));
        }
    }
    return acc;
}

// Automatic lanes per scored item (vertex, candidate or proposal): about ten
// partitions per lane for the largest k of the context.  Fewer lanes per item
// means more items per warp and fewer group reductions; timed on GB300 over
// 1..32 lanes, this was fastest for k = 20 (2 lanes) and k = 50 (8 lanes).
__host__ __device__ __forceinline__ int lanes_per_item(int k)
{
    int gs = 1;
    while (gs < 32 && gs * 10 < k) gs <<= 1;
    return gs;
}

// ---- A_a of the own cluster ------------------------------------------
// own[v] = {A_a, change stamp of a when it was computed}.  A_a is a function
// of v's cluster alone, so it holds until a move into or out of that cluster
// (which stamps it, chg[]).  A heavy sweep computes it for every vertex
// whose cluster changed (h_eval: in the order of the member list, so that a
// cluster's summary row or its members' rows stay in L1, and their sum is the
// table part of F'); any other vertex computes it when it has a candidate to
// score (edges), so vertices whose neighbours all share their cluster cost
// nothing.
__device__ __forceinline__ bool own_valid(int2 o, int chg)
{
    return o.y >= chg;
}

// This lane's share of A_c(v) for a member v of cluster c (size sc).
__device__ __forceinline__ int own_part(const SweepArgs& a, const JobInfo& J, unsigned long long mask, int small,
                                        long long v, int c, int sc, int l, int gs)
{
    const int* gv = a.G + row_of(J, v);
    if (sc == 1) return l == 0 ? J.k : 0;
    if (sc <= small) return member_part(a, J, gv, c, sc, l, gs);
    int ex = 0, ub = 0;
    summary_part(a, J, gv, c, sc, l, gs, ex, ub);
    return ex + probe_part(a, J, a.table, mask, gv, c, sc, l, gs);
}

// ---- active set ------------------------------------------------------
// With cc_options.active_set, every move stamps its two clusters with the
// sweep's number, and a sweep after the first of a run re-scores only what
// the previous sweep can have changed.  v's gain towards a candidate x
// depends on A_a and |a| of its own cluster a and on |x| and A_x of x; v's
// candidates are the clusters of its neighbours, and a neighbour that moves
// stamps both its clusters.  So:
//   * if neither a nor the target of v's previous bid was stamped, the
//     candidates that were not stamped keep their gains, and v's new bid is
//     the least of its previous bid and the bids of its stamped candidates:
//     only those are scored;
//   * otherwise (act[v] = 1) every candidate of v is scored.
// The first sweep of a run scores everything.

// Per-vertex part of the proposal step that the options need: the active
// set's flags, and the bid of the move-to-empty variant (a group of lanes per
// vertex).  Nothing to do without those options.
// kSingle: the context holds one job, so every vertex belongs to job 0 and
// the job is running whenever the sweep is not skipped.
template <bool kSingle>
__device__ __forceinline__ void own_phase(const SweepArgs& a)
{
    DevState* st = a.st;
    if (st->skip || (!a.active_set && !a.empty_moves)) return;
    const unsigned long long mask = st->mask;
    const int gs = a.gs, small = st->small;
    const int lane = threadIdx.x & 31, l = lane & (gs - 1);
    const long long groups = (long long)gridDim.x * blockDim.x / gs;
    const JobInfo J0 = first_job(a);
    const int all = st->all_active, last = st->stamp - 1;
    // colour_batched: only the vertices of the current class, listed in vlist
    long long count = a.n, vbase = 0;
    if (a.colour_mode) {
        vbase = a.voff[st->cls];
        count = a.voff[st->cls + 1] - vbase;
    }
    for (long long base = ((long long)blockIdx.x * blockDim.x + threadIdx.x - lane) / gs; base < count;
         base += groups) {
        const long long idx = base + lane / gs;
        const bool valid = idx < count;
        const long long v = a.colour_mode ? (valid ? (long long)__ldg(a.vlist + vbase + idx) : 0) : idx;
        const int j = (kSingle || !valid) ? 0 : __ldg(a.jid + v);
        const bool run = valid && (kSingle || !a.js[j].stop);
        const int cv = run ? a.C[v] : 0;
        if (a.active_set && run && l == 0) {
            // active set: every candidate again if a or the previous bid's
            // target changed
            const unsigned long long p = a.prev[v];
            const bool full = all || a.chg[cv] == last ||
                              (p != kEmpty && a.chg[(int)(unsigned)(p & 0xffffffffull)] == last);
            a.act[v] = full ? 1 : 0;
        }
        // move-to-empty variant: the empty cluster with id v is a candidate
        // while no vertex carries that id (sizes are those of the sweep start)
        const bool iso = a.empty_moves && run && a.size[v] == 0;
        if (!__any_sync(kFull, iso)) continue;
        const JobInfo J = kSingle ? J0 : a.job[j];
        const int chg = iso ? a.chg[cv] : 0, sa = iso ? a.size[cv] : 1;
        const int2 o = iso ? a.own[v] : make_int2(0, 0);
        int part = 0;
        if (iso && !own_valid(o, chg)) part = own_part(a, J, mask, small, v, cv, sa, l, gs);
        const int A = group_sum(part, gs);
        if (iso && l == 0) {
            if (!own_valid(o, chg)) a.own[v] = make_int2(A, chg);
            // Eq. objective3 with an empty target: 2 (A_a - k) - k (|a| - 1)
            const int Aa = own_valid(o, chg) ? o.x : A;
            const int dD = 2 * (Aa - J.k) - J.k * (sa - 1);
            if (dD < 0) atomicMin(&a.best[v], pack_key(dD, (int)v));
        }
    }
}

// One window of CSR entries of one warp in shared memory: kChunks chunks of
// 32 entries are gathered before scoring, so that the scoring rounds (32 / gs
// candidates each) run nearly full.  Candidates: singletons from the front,
// other clusters from the back.  Slots: the distinct vertices of the window,
// kSlots of them scored at a time (more in one window are rare).  The size
// matters: four blocks' scratch (29 KB each) leave 96 KB of the SM's memory to
// the L1 that the gathers of rows go through; at 40 KB (64 KB of L1) the step
// took 7% longer, with no L1 to speak of 54%.
constexpr int kChunks = 4;
constexpr int kSpan = 32 * kChunks;
constexpr int kSlots = 64;
static_assert(16 * kSmall <= kSpan, "the pairs of 16 small candidates must fit the scratch");
struct EdgeScratch {
    unsigned long long ubest[kSlots];  // slot: upper bound on the vertex's final bid
    int base[kSlots];                  //   2 (A_a - k) - k (|a| - 1), so dD = base + k |x| - 2 A_x
    int v[kSpan];                      // vertex of each slot of the window
    int x[kSpan];                      // candidate: cluster,
    int w[kSpan];                      //   its size (singleton: its vertex),
    int lo[kSpan];                     //   least dD.  Before that: the clusters of the slots, then each slot's
                                       //   largest candidate (|x| << 7 | index); small clusters: members of the pairs
    int part[kSpan];                   //   exact part of A_x
    unsigned char slot[kSpan];         //   its slot, | 128 if it is its vertex's largest
    unsigned char list[kSpan], pair[kSpan];
};

// The proposal step's scoring.  CSR entries 32 at a time per warp: each lane
// reads one entry (v, u) and keeps it if v's job runs and u lies in another
// cluster than v (self-loops and repeats of the same (v, C[u]) inside the 32
// entries are dropped).  The candidates kept from kChunks chunks are scored
// by groups of lanes, in an order that leaves little to score:
//   1. A_a of each vertex with a candidate (own[], or computed now);
//   2. each vertex's largest candidate: with A_x at its bound k |x| the
//      larger cluster has the lower possible dD, so its dD is a good bound;
//   3. the other candidates whose packed (least dD at A_x = k |x|, x) is
//      below the vertex's bound so far, compacted into full rounds;
//   4. of those, hash probes where the summary leaves partitions open and the
//      summary's least dD is still below the bound;
//   5. singletons below the bound: two label rows compared.
// A candidate that is skipped cannot be its vertex's least bid (its packed
// least dD is not below an upper bound on it), and one whose dD cannot be
// negative is never proposed, so the bids, and the proposals, do not depend
// on what was skipped.  On kNN graphs (n = 1e5, k = 50) step 2 leaves 11.4
// of 19.0 candidates per vertex in sweep 2 and 3.5 of 6.0 in sweep 3.
// Clusters of at most st->small members are scored from their members' rows,
// larger ones from their summary rows and probes.  A move with dD < 0 bids
// its packed (dD, x) at best[v] with an atomic minimum.  All group reductions
// are outside the branches, so every lane takes part in every shuffle.  sh:
// the block's scratch in shared memory, one per warp.
template <bool kSingle>
__device__ __forceinline__ void edges_phase(const SweepArgs& a, EdgeScratch* sh)
{
    DevState* st = a.st;
    if (st->skip) return;
    const unsigned long long mask = st->mask;
    const int gs = a.gs, per = 32 / gs, small = st->small;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, l = lane & (gs - 1), grp = lane / gs;
    const unsigned lt = (1u << lane) - 1u;
    EdgeScratch& es = sh[w];
    const JobInfo J0 = first_job(a);
    // row compares (a plain streaming compare) take half the lanes, an eighth with
    // 16-bit rows (k = 50: 24.05 ms with half, 22.63 with a quarter, 22.54 so)
    const int gr = max(1, gs >> (kSingle && !J0.narrow ? 1 : 3)), pr = 32 / gr, lr = lane & (gr - 1);
    const int all = st->all_active, last = st->stamp - 1;
    const bool many = st->many != 0;
    // colour_batched: only the CSR entries of the current class's vertices,
    // listed in eidx
    const int* eidx = nullptr;
    long long count = a.nnz;
    if (a.colour_mode) {
        const long long e0 = a.eoff[st->cls];
        eidx = a.eidx + e0;
        count = a.eoff[st->cls + 1] - e0;
    }
    // entries of a window: fewer than kSpan where that leaves warps idle (a
    // small job, a colour class), for the window's latency is then the step's
    const unsigned nwarps = gridDim.x * kWarpsPerBlock;
    const int span = count >= (long long)kSpan * nwarps
                         ? kSpan
                         : 32 * (int)max(1LL, min((long long)kChunks, (count + 32 * nwarps - 1) / (32 * nwarps)));
    const long long windows = (count + span - 1) / span;
    __shared__ int s_taken;
    const WarpQueue queue{&s_taken};
    queue.start();
    for (long long win = queue.next(); win < windows; win = queue.next()) {
        int ns = 0, nt = 0, slots = 0;
        // the loads of all kChunks chunks first (entries, then clusters, then
        // sizes), so that their latencies overlap; then each chunk's votes
        // and compaction
        int vc[kChunks], uc[kChunks], xc[kChunks], sc[kChunks];
#pragma unroll
        for (int c = 0; c < kChunks; ++c) {
            const long long ep = win * span + c * 32 + lane;
            vc[c] = -1;
            uc[c] = -1;
            if (ep < count && c * 32 < span) {
                const long long e = eidx ? (long long)__ldg(eidx + ep) : ep;
                vc[c] = __ldg(a.src + e);
                uc[c] = __ldg(a.col + e);
            }
        }
#pragma unroll
        for (int c = 0; c < kChunks; ++c) {
            xc[c] = -1;
            sc[c] = -1;
            if (uc[c] != vc[c] && (kSingle || !a.js[__ldg(a.jid + vc[c])].stop)) {
                xc[c] = a.C[uc[c]];
                sc[c] = a.C[vc[c]];
            }
        }
#pragma unroll
        for (int c = 0; c < kChunks; ++c) {
            es.part[c * 32 + lane] = sc[c];  // the vertex's cluster, for its slot
            if (xc[c] == sc[c]) xc[c] = -1;
            // active set: only candidates that changed, unless v is scored in full
            if (xc[c] >= 0 && a.active_set && !all && !a.act[vc[c]] && a.chg[xc[c]] != last) xc[c] = -1;
            sc[c] = xc[c] >= 0 ? a.size[xc[c]] : 0;
        }
        int before = -1;  // vertex of the kept entry before the chunk
#pragma unroll
        for (int c = 0; c < kChunks; ++c) {
            const int v = vc[c], x = xc[c], sx = sc[c];
            if (!__any_sync(kFull, x >= 0)) continue;
            // entries of one vertex are contiguous: from is the first lane of
            // v's entries in the chunk, and v's entries before this lane are
            // those from there on
            const int up = __shfl_up_sync(kFull, v, 1);
            const unsigned starts = __ballot_sync(kFull, lane == 0 || up != v);
            const unsigned mine = lt & (~0u << (31 - __clz(starts & (lt | (1u << lane)))));
            const unsigned same = __match_any_sync(kFull, x);
            const bool keep = x >= 0 && !(same & mine);
            const unsigned kept = __ballot_sync(kFull, keep);
            // a vertex's first kept entry opens its slot
            const bool head = keep && !(kept & mine) && v != before;
            const unsigned heads = __ballot_sync(kFull, head);
            const int slot = slots + __popc(heads & (lt | (1u << lane))) - 1;
            if (head) {
                es.v[slot] = v;
                es.lo[slot] = es.part[c * 32 + lane];
            }
            slots += __popc(heads);
            before = __shfl_sync(kFull, v, 31 - __clz(kept));
            const bool sgl = keep && sx == 1;
            const unsigned ks = __ballot_sync(kFull, sgl), kt = kept & ~ks;
            if (keep) {
                const int p = sgl ? ns + __popc(ks & lt) : kSpan - 1 - (nt + __popc(kt & lt));
                es.x[p] = x;
                es.w[p] = sgl ? uc[c] : sx;
                es.slot[p] = (unsigned char)slot;
            }
            ns += __popc(ks);
            nt += __popc(kt);
        }
        __syncwarp();
        if (slots == 0) continue;
        for (int sb = 0; sb < slots; sb += kSlots) {
            const int count_s = min(slots - sb, kSlots);
            auto in_batch = [&](int f) { return ((f & 127) & ~(kSlots - 1)) == sb; };
            // A_a per slot: a lane per slot reads what is known; the rest is
            // computed by groups of lanes
            for (int s0 = 0; s0 < count_s; s0 += 32) {
                const int s = s0 + lane;
                bool stale = false;
                int v = 0, cv = 0, chg = 0, sa = 1;
                if (s < count_s) {
                    v = es.v[sb + s];
                    cv = sb == 0 ? es.lo[s] : a.C[v];  // (the later slots' clusters have been overwritten)
                    const int2 o = a.own[v];
                    chg = a.chg[cv];
                    sa = a.size[cv];
                    const unsigned long long b0 = __ldcg(a.best + v);
                    const int k = kSingle ? J0.k : a.job[__ldg(a.jid + v)].k;
                    stale = !own_valid(o, chg);
                    es.base[s] = 2 * (o.x - k) - k * (sa - 1);
                    es.ubest[s] = b0;
                }
                unsigned todo = __ballot_sync(kFull, stale);
                __syncwarp();
                if (s < count_s) es.lo[s] = 0;
                while (todo) {
                    // the group's slot: the grp-th stale one
                    unsigned t = todo;
                    for (int i = 0; i < grp; ++i) t &= t - 1;
                    const bool on = t != 0;
                    const int q = on ? __ffs(t) - 1 : lane;
                    const int vq = __shfl_sync(kFull, v, q), cq = __shfl_sync(kFull, cv, q);
                    const int sq = __shfl_sync(kFull, sa, q), hq = __shfl_sync(kFull, chg, q);
                    const JobInfo J = kSingle ? J0 : a.job[__ldg(a.jid + vq)];
                    int part = 0;
                    if (on) part = own_part(a, J, mask, small, vq, cq, sq, l, gs);
                    part = group_sum(part, gs);
                    if (on && l == 0) {
                        a.own[vq] = make_int2(part, hq);
                        es.base[s0 + q] = 2 * (part - J.k) - J.k * (sq - 1);
                    }
                    for (int i = 0; i < per && todo; ++i) todo &= todo - 1;
                }
            }
            __syncwarp();
            // the largest candidate of each slot
            if (many) {
                for (int c0 = 0; c0 < nt; c0 += 32) {
                    const int q = kSpan - 1 - (c0 + lane);
                    if (c0 + lane < nt && in_batch(es.slot[q]))
                        atomicMax(reinterpret_cast<unsigned*>(&es.lo[es.slot[q] & (kSlots - 1)]),
                                  ((unsigned)es.w[q] << 7) | (unsigned)q);
                }
                __syncwarp();
                for (int c0 = 0; c0 < nt; c0 += 32) {
                    const int q = kSpan - 1 - (c0 + lane);
                    if (c0 + lane < nt && in_batch(es.slot[q]) && (es.lo[es.slot[q] & (kSlots - 1)] & 127) == q)
                        es.slot[q] |= 128;
                }
                __syncwarp();
            }
            // the clusters: the largest ones first, then the others (all at once
            // when few vertices moved in the sweep before: the bounds then rule
            // out little)
            for (int pass = many ? 0 : 1; pass < 2; ++pass) {
                // list: candidates above `small` from the front, others from the back
                int nl = 0, nm = 0;
                for (int c0 = 0; c0 < nt; c0 += 32) {
                    const int q = kSpan - 1 - (c0 + lane);
                    bool on = c0 + lane < nt, big = true;
                    if (on) {
                        const int f = es.slot[q], s = f & (kSlots - 1), sx = es.w[q];
                        const int k = kSingle ? J0.k : a.job[__ldg(a.jid + es.v[f & 127])].k;
                        // A_x <= k |x|
                        const int lo = es.base[s] - k * sx;
                        on = in_batch(f) && (!many || (f >= 128) == (pass == 0)) && lo < 0 &&
                             pack_key(lo, es.x[q]) < es.ubest[s];
                        big = sx > small;
                    }
                    const unsigned bb = __ballot_sync(kFull, on && big), bm = __ballot_sync(kFull, on && !big);
                    if (on) {
                        const int p = big ? nl + __popc(bb & lt) : kSpan - 1 - (nm + __popc(bm & lt));
                        es.list[p] = (unsigned char)q;
                    }
                    nl += __popc(bb);
                    nm += __popc(bm);
                }
                __syncwarp();
                // small clusters: every (candidate, member) pair is one row
                // compare, 16 candidates at a time (at most 16 kSmall pairs), so
                // that the rounds run full and no load waits for another
                for (int c0 = 0; c0 < nm; c0 += 16) {
                    const bool mine = lane < 16 && c0 + lane < nm;
                    const int q = mine ? (int)es.list[kSpan - 1 - (c0 + lane)] : 0;
                    const int sx = mine ? es.w[q] : 0;
                    int end = sx;  // pairs up to and including this lane's
                    for (int o = 1; o < 16; o <<= 1) {
                        const int y = __shfl_up_sync(kFull, end, o);
                        if (lane >= o) end += y;
                    }
                    const int pairs = __shfl_sync(kFull, end, 15);
                    if (mine) {
                        const int* mem = a.members + (a.cursor[es.x[q]] - sx);
                        es.part[q] = 0;
                        for (int m = 0; m < sx; ++m) {
                            es.lo[end - sx + m] = mem[m];
                            es.pair[end - sx + m] = (unsigned char)q;
                        }
                    }
                    __syncwarp();
                    for (int r0 = 0; r0 < pairs; r0 += pr) {
                        const bool valid = r0 + lane / gr < pairs;
                        const int p = valid ? r0 + lane / gr : 0;
                        const int pq = es.pair[p], v = es.v[es.slot[pq] & 127];
                        const JobInfo J = kSingle ? J0 : a.job[__ldg(a.jid + v)];
                        int part = 0;
                        if (valid) part = same_part(a, J, es.lo[p], v, lr, gr);
                        part = group_sum(part, gr);
                        if (valid && lr == 0) atomicAdd(&es.part[pq], part);
                    }
                    __syncwarp();
                    if (mine) {
                        const int v = es.v[es.slot[q] & 127], s = es.slot[q] & (kSlots - 1), x = es.x[q];
                        const int k = kSingle ? J0.k : a.job[__ldg(a.jid + v)].k;
                        const int dD = es.base[s] + k * sx - 2 * es.part[q];
                        const unsigned long long key = pack_key(dD, x);
                        if (dD < 0 && key < es.ubest[s]) {
                            atomicMin(&es.ubest[s], key);
                            atomicMin(&a.best[v], key);
                        }
                    }
                    __syncwarp();
                }
                // larger clusters: their summary rows
                int no = 0;  // left open by the summary
                for (int r0 = 0; r0 < nl; r0 += per) {
                    const bool valid = r0 + grp < nl;
                    const int q = valid ? (int)es.list[r0 + grp] : 0;
                    const int f = valid ? (int)es.slot[q] : 0, s = f & (kSlots - 1);
                    const int v = valid ? es.v[f & 127] : 0, x = valid ? es.x[q] : 0, sx = valid ? es.w[q] : 0;
                    const JobInfo J = kSingle ? J0 : a.job[valid ? __ldg(a.jid + v) : 0];
                    int part = 0, ub = 0;
                    if (valid) summary_part(a, J, a.G + row_of(J, v), x, sx, l, gs, part, ub);
                    part = group_sum(part, gs);
                    ub = group_sum(ub, gs);
                    bool open = false;
                    if (valid && l == 0) {
                        const int top = es.base[s] + J.k * sx;  // dD = top - 2 A
                        const int lo = top - 2 * ub, hi = top - 2 * part;
                        const unsigned long long key = pack_key(hi, x);
                        if (hi < 0 && key < es.ubest[s]) atomicMin(&es.ubest[s], key);
                        if (ub == part) {
                            if (hi < 0 && key <= es.ubest[s]) atomicMin(&a.best[v], key);
                        } else if (lo < 0) {
                            es.lo[q] = lo;
                            es.part[q] = part;
                            open = true;
                        }
                    }
                    // the list entries of this round are read already: the open
                    // ones go back to the front
                    const unsigned bal = __ballot_sync(kFull, open);
                    __syncwarp();
                    if (open) es.list[no + __popc(bal & lt)] = (unsigned char)q;
                    no += __popc(bal);
                }
                __syncwarp();
                // probes of the open ones still below the bound, in full rounds
                int np = 0;
                for (int c0 = 0; c0 < no; c0 += 32) {
                    const int q = c0 + lane < no ? (int)es.list[c0 + lane] : 0;
                    const bool on = c0 + lane < no && pack_key(es.lo[q], es.x[q]) < es.ubest[es.slot[q] & (kSlots - 1)];
                    const unsigned bal = __ballot_sync(kFull, on);
                    __syncwarp();
                    if (on) es.list[np + __popc(bal & lt)] = (unsigned char)q;
                    np += __popc(bal);
                }
                __syncwarp();
                for (int r0 = 0; r0 < np; r0 += per) {
                    const bool valid = r0 + grp < np;
                    const int q = valid ? (int)es.list[r0 + grp] : 0;
                    const int f = valid ? (int)es.slot[q] : 0, s = f & (kSlots - 1);
                    const int v = valid ? es.v[f & 127] : 0, x = valid ? es.x[q] : 0, sx = valid ? es.w[q] : 0;
                    const JobInfo J = kSingle ? J0 : a.job[valid ? __ldg(a.jid + v) : 0];
                    int pb = 0;
                    if (valid) pb = probe_part(a, J, a.table, mask, a.G + row_of(J, v), x, sx, l, gs);
                    pb = group_sum(pb, gs);
                    if (valid && l == 0) {
                        const int dD = es.base[s] + J.k * sx - 2 * (es.part[q] + pb);
                        const unsigned long long key = pack_key(dD, x);
                        if (dD < 0 && key <= es.ubest[s]) {
                            atomicMin(&es.ubest[s], key);
                            atomicMin(&a.best[v], key);
                        }
                    }
                }
                __syncwarp();
            }
            // singletons
            int nl = 0;
            for (int c0 = 0; c0 < ns; c0 += 32) {
                const int q = c0 + lane;
                bool on = q < ns;
                if (on) {
                    const int f = es.slot[q], s = f & (kSlots - 1);
                    const int k = kSingle ? J0.k : a.job[__ldg(a.jid + es.v[f])].k;
                    const int lo = es.base[s] - k;
                    on = in_batch(f) && lo < 0 && pack_key(lo, es.x[q]) < es.ubest[s];
                }
                const unsigned bal = __ballot_sync(kFull, on);
                if (on) es.list[nl + __popc(bal & lt)] = (unsigned char)q;
                nl += __popc(bal);
            }
            __syncwarp();
            for (int r0 = 0; r0 < nl; r0 += pr) {
                const bool valid = r0 + lane / gr < nl;
                const int q = valid ? (int)es.list[r0 + lane / gr] : 0;
                const int f = valid ? (int)es.slot[q] : 0, s = f & (kSlots - 1);
                const int v = valid ? es.v[f] : 0;
                const JobInfo J = kSingle ? J0 : a.job[valid ? __ldg(a.jid + v) : 0];
                int part = 0;
                if (valid) part = same_part(a, J, es.w[q], v, lr, gr);
                part = group_sum(part, gr);
                if (valid && lr == 0) {
                    const int dD = es.base[s] + J.k - 2 * part;
                    const unsigned long long key = pack_key(dD, es.x[q]);
                    if (dD < 0 && key < es.ubest[s]) {
                        atomicMin(&es.ubest[s], key);
                        atomicMin(&a.best[v], key);
                    }
                }
            }
            __syncwarp();
        }
    }
}

// Turns the bids into the proposal list (v, a, b, dD), counts them per job and
// clears best[].  A block takes tiles of one vertex per thread, or of four
// where that still gives every block one, and one range of the list per tile:
// adds to the list's length go through one after another, about 6 ns each, and
// were most of the step with small tiles and a sum per warp for the job's
// count (n = 1e6: 22 us; with fewer tiles than blocks, n = 1.5e5, large ones
// took 13 us instead of 11).  With one job the length is the job's count, and
// route_phase copies it.
__device__ __forceinline__ void collect_phase(const SweepArgs& a)
{
    constexpr int kPer = 4;
    extern __shared__ long long dyn_jobs[];
    DevState* st = a.st;
    if (st->skip) return;
    __shared__ int s_cnt, s_keys;
    __shared__ unsigned long long s_base;
    const bool many_jobs = a.jobs > 1;
    JobAcc acc(job_smem_init(a.jobs, dyn_jobs), reinterpret_cast<long long*>(&a.js[0].nprop), kJobStride);
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const int per = a.n >= (long long)gridDim.x * (kPer * kBlock) ? kPer : 1;
    const long long stride = (long long)gridDim.x * (per * kBlock);
    for (long long b0 = (long long)blockIdx.x * (per * kBlock) + threadIdx.x; b0 - threadIdx.x < a.n; b0 += stride) {
        if (threadIdx.x == 0) {
            s_cnt = 0;
            s_keys = 0;
        }
        __syncthreads();
        unsigned long long key[kPer];
        int rank[kPer], total = 0, keys = 0;
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            const long long v = b0 + q * kBlock;
            key[q] = q < per && v < a.n ? a.best[v] : kEmpty;
        }
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            const long long v = b0 + q * kBlock;
            if (q > 0 && q >= per) break;
            if (key[q] != kEmpty) a.best[v] = kEmpty;
            if (a.active_set && v < a.n) {
                // a vertex scored only on its changed candidates keeps its
                // previous bid if that is still the least; a vertex of a
                // stopped job bids nothing
                if (a.js[a.jid[v]].stop) key[q] = kEmpty;
                else if (!st->all_active && !a.act[v] && a.prev[v] < key[q]) key[q] = a.prev[v];
                a.prev[v] = key[q];
            }
            const unsigned on = __ballot_sync(kFull, key[q] != kEmpty);
            rank[q] = total + __popc(on & lt);
            total += __popc(on);
            if (many_jobs && key[q] != kEmpty) {
                const int job = a.jid[v];
                acc.add(job, 1);
                keys += a.job[job].k;
            }
        }
        if (many_jobs)
            for (int o = 16; o > 0; o >>= 1) keys += __shfl_xor_sync(kFull, keys, o);
        int base = 0;
        if (lane == 0 && total) {
            base = atomicAdd(&s_cnt, total);
            if (many_jobs) atomicAdd(&s_keys, keys);
        }
        base = __shfl_sync(kFull, base, 0);
        __syncthreads();
        if (threadIdx.x == 0 && s_cnt > 0) {
            s_base = atomicAdd(&st->nprop, (unsigned long long)s_cnt);
            if (many_jobs) atomicAdd(&st->pkeys, (unsigned long long)s_keys);
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kPer; ++q)
            if (key[q] != kEmpty) {
                const long long v = b0 + q * kBlock;
                const unsigned long long p = s_base + (unsigned)(base + rank[q]);
                a.pv[p] = (int)v;
                a.pa[p] = a.C[v];
                a.pb[p] = (int)(unsigned)(key[q] & 0xffffffffull);
                a.pg[p] = key_gain(key[q]);
            }
    }
    if (many_jobs) job_acc_finish(acc, a.jobs);
}

// ---- heavy sweeps --------------------------------------------------------
// When the proposals move a large share of the label rows (more than 1/8 of
// sum_j k_j n_j; for one job |P| > n / 8), or always with sweep_mode 2, never
// with sweep_mode 1, or when the table does not hold the
// counts of C yet (the singleton start), dF(P1) is taken from a rebuild
// instead of from staged deltas: P1 is applied to C in place (the movers' old
// clusters stay in the proposal list), the table and its summary rows are
// rebuilt from the new C, and F' - F is dF(P1) exactly for every job.  A job
// whose dF is negative has committed P1 (mode 3); any other job's moves are
// undone, the table is rebuilt from C again and its matching fallback runs as
// in a light sweep (mode 2).

__device__ __forceinline__ void route_phase(const SweepArgs& a)
{
    const unsigned long long total_keys = a.keys;
    DevState* st = a.st;
    st->heavy = 0;
    if (st->skip) return;
    if (a.jobs == 1) {
        a.js[0].nprop = st->nprop;
        st->pkeys = st->nprop * (unsigned long long)a.job[0].k;
    }
    if (st->err || st->nprop == 0) return;
    // light when the proposals move at most 1/8 of all label rows (for one
    // job: |P| <= n / 8)
    const bool light = a.sweep_mode == 1 || (a.sweep_mode == 0 && st->pkeys * 8 <= total_keys);
    if (st->tvalid && !st->small && light) return;
    st->heavy = 1;
    // keys after applying P1: every vertex gives at most k, every mover at most k new ones
    unsigned long long bound = (!st->tvalid ? total_keys : st->small ? st->keys_all : (unsigned long long)st->live) +
                               st->pkeys;
    if (bound > total_keys) bound = total_keys;
    unsigned long long c = a.cap_min;
    while (c < 2 * bound && c < a.mask_max + 1) c <<= 1;
    st->safe_mask = c - 1;
    // the capacity of the rebuild is settled once the sizes after P1 are
    // known (size_build)
    st->build_light = light ? 1 : 0;
    st->build_small = 0;
    st->small_keys = 0;
    st->sized = 0;
    st->new_mask = c - 1;
    st->retry_mask = c - 1;
    st->rebuild = 1;
}

// Singleton guard on every proposal (sizes of the sweep start); counts |P1| per job.
__device__ __forceinline__ void h_mark_phase(const SweepArgs& a)
{
    extern __shared__ long long dyn_jobs[];
    DevState* st = a.st;
    if (st->skip || !st->heavy) return;
    JobAcc acc(job_smem_init(a.jobs, dyn_jobs), reinterpret_cast<long long*>(&a.js[0].np1), kJobStride);
    const long long np = (long long)st->nprop;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < np; p += stride) {
        const int ca = a.pa[p], cb = a.pb[p];
        const bool keep = !(a.size[ca] == 1 && a.size[cb] == 1) || cb < ca;
        a.pflag[p] = keep ? 1 : 0;
        if (keep) acc.add(a.jid[a.pv[p]], 1);
    }
    job_acc_finish(acc, a.jobs);
}

// Applies (undo = 0) or undoes (undo = 1, jobs that roll back only) the kept
// proposals on C and the sizes.
__device__ __forceinline__ void h_apply_phase(const SweepArgs& a, int undo)
{
    DevState* st = a.st;
    if (st->skip || !st->heavy || (undo && !st->rollback)) return;
    const long long np = (long long)st->nprop;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < np; p += stride) {
        if (!a.pflag[p]) continue;
        const int v = a.pv[p];
        if (undo && !a.js[a.jid[v]].rollback) continue;
        const int ca = a.pa[p], cb = a.pb[p];
        a.C[v] = undo ? ca : cb;
        atomicAdd(&a.size[ca], undo ? 1 : -1);
        atomicAdd(&a.size[cb], undo ? -1 : 1);
        if (!undo) {
            a.chg[ca] = st->stamp;
            a.chg[cb] = st->stamp;
        }
    }
}

// F' per job after P1: k sum_c s_c^2 - 2 sum_v A_c(v)(v), since the counts of a
// cluster's label classes, squared, are the sum of A_c over its members.  A_a
// is computed for every vertex whose cluster changed (and kept for the next
// sweep), in the order of the member list, 32 members of a warp at a time.
// Members of one cluster follow each other, so its summary row is read from
// L1 after the first.  With a partial table the clusters without summary rows
// are counted inside the warp: each lane reads its member's label row once,
// and the lanes of its cluster with the same label are its count.  Windows
// then overlap by kSmall, so that a small cluster lies whole in the window
// that holds its first member.
template <bool kSingle>
__device__ __forceinline__ void h_eval_phase(const SweepArgs& a)
{
    extern __shared__ long long dyn_jobs[];
    DevState* st = a.st;
    if (st->skip || !st->heavy || st->err || st->again) return;
    JobAcc acc(job_smem_init(a.jobs, dyn_jobs), &a.js[0].recompute, kJobStride);
    const unsigned long long mask = st->new_mask;
    const int gs = a.gs, per = 32 / gs, small = st->build_small;
    const int lane = threadIdx.x & 31, l = lane & (gs - 1), grp = lane / gs;
    const int step = 32 - small;
    const JobInfo J0 = first_job(a);
    __shared__ int s_taken;
    const WarpQueue queue{&s_taken};
    queue.start();
    for (long long wb = queue.next() * step; wb < a.n; wb = queue.next() * step) {
        const long long idx = wb + lane;
        const int v = idx < a.n ? a.members[idx] : 0;
        // (a place holding a smaller job leaves vertices to the idle job)
        bool valid = idx < a.n && (!kSingle || v < J0.n);
        const int c = valid ? a.C[v] : -1 - lane;
        const int sc = valid ? a.size[c] : 1, chg = valid ? a.chg[c] : 0, end = valid ? a.cursor[c] : 0;
        const int2 o = valid ? a.own[v] : make_int2(0, 0);
        const int job = (kSingle || !valid) ? 0 : __ldg(a.jid + v);
        const int k = kSingle ? J0.k : a.job[job].k;
        const bool in_warp = valid && sc > 1 && sc <= small;
        // a small cluster belongs to the window of its first member, any
        // other member to the window that steps over it
        const long long at = in_warp ? end - sc : idx;
        valid = valid && at >= wb && at < wb + step;
        const bool known = !valid || sc == 1 || own_valid(o, chg);
        int A = sc == 1 ? k : o.x;
        const bool count = valid && in_warp;
        if (__any_sync(kFull, count && !known)) {
            // lanes of this lane's cluster (all of them in the window, and
            // all of them counted, whether or not their own sum is known)
            const unsigned lanes = count ? (~0u >> (32 - sc)) << (int)(at - wb) : 0u;
            const int4* row = reinterpret_cast<const int4*>(a.G + row_of(kSingle ? J0 : a.job[job], valid ? v : 0));
            int sum = 0;
            for (int i = 0; i < a.kmax; i += 4) {
                int4 g = make_int4(-1, -1, -1, -1);
                if (count && i < k) g = __ldg(row + (i >> 2));
                sum += __popc(__match_any_sync(kFull, g.x) & (i < k ? lanes : 0u));
                if (i + 1 < a.kmax) sum += __popc(__match_any_sync(kFull, g.y) & (i + 1 < k ? lanes : 0u));
                if (i + 2 < a.kmax) sum += __popc(__match_any_sync(kFull, g.z) & (i + 2 < k ? lanes : 0u));
                if (i + 3 < a.kmax) sum += __popc(__match_any_sync(kFull, g.w) & (i + 3 < k ? lanes : 0u));
            }
            if (count && !known) A = sum;
        }
        // the others: a group of lanes per member
        unsigned todo = __ballot_sync(kFull, valid && !known && !in_warp);
        while (todo) {
            unsigned t = todo;
            for (int i = 0; i < grp; ++i) t &= t - 1;
            const bool on = t != 0;
            const int q = on ? __ffs(t) - 1 : lane;
            const int vq = __shfl_sync(kFull, v, q), cq = __shfl_sync(kFull, c, q), sq = __shfl_sync(kFull, sc, q);
            const JobInfo J = kSingle ? J0 : a.job[__shfl_sync(kFull, job, q)];
            int part = 0;
            if (on) part = own_part(a, J, mask, 0, vq, cq, sq, l, gs);
            part = group_sum(part, gs);
            // back to the members' lanes: the i-th of todo was group i's
            const unsigned round = todo;
            int left = per;
            for (; left > 0 && todo; --left) todo &= todo - 1;
            const unsigned done = round & ~todo;
            const int from = __popc(done & ((1u << lane) - 1u)) * gs;
            const int got = __shfl_sync(kFull, part, from & 31);
            if (done >> lane & 1u) A = got;
        }
        if (valid) {
            if (!known) a.own[v] = make_int2(A, chg);
            else if (sc == 1) a.own[v] = make_int2(k, chg);
            // each member adds its share k s of its cluster's k s^2
            acc.add(job, (long long)k * sc - 2LL * A);
        }
    }
    job_acc_finish(acc, a.jobs);
}

__device__ __forceinline__ void h_decide_phase(const SweepArgs& a, int t0, int stride)
{
    DevState* st = a.st;
    if (st->skip || !st->heavy) return;
    for (int j = t0; j < a.jobs; j += stride) {
        JobState& s = a.js[j];
        if (s.stop) continue;
        if (st->err) {
            s.mode = 0;
            continue;
        }
        const long long dF = s.recompute + s.partition_sq - s.F;
        s.dF_p1 = s.np1 > 0 ? dF : 0;
        if (s.np1 > 0 && dF < 0) {
            s.mode = 3;
            s.dF = dF;
            s.moves = s.np1;
        } else {
            s.mode = s.nprop > 0 ? 2 : 0;
            if (s.mode == 2) st->match = 1;
            s.dF = 0;
            s.moves = 0;
            if (s.np1 > 0) s.rollback = 1;
            // the rollback rebuilds at the capacity that holds every key the
            // sweep can create, so that the matching fallback's inserts fit;
            // a job that falls back without moves to undo also needs that
            // room when the heavy rebuild was a tight one
            if (s.np1 > 0 || (s.mode == 2 && (st->mask != st->safe_mask || st->small))) {
                st->rollback = 1;
                st->rebuild = 1;
                st->new_mask = st->safe_mask;
                st->build_small = 0;  // the matching needs every key
            }
        }
    }
}

// ---- light sweeps -------------------------------------------------------

// Occupancy above which a sweep is abandoned and retried in a larger table.
__device__ __forceinline__ unsigned long long fill_limit(unsigned long long mask)
{
    return (mask + 1) - ((mask + 1) >> 3);
}

// Adds the warp's new slots to st->used and flags an overflow past the limit.
// All lanes must call it.
__device__ __forceinline__ void count_inserts(DevState* st, int mine, unsigned long long mask)
{
    int x = mine;
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
    if ((threadIdx.x & 31) == 0 && x > 0) {
        const unsigned long long old = atomicAdd(&st->used, (unsigned long long)x);
        if (old + x > fill_limit(mask)) st->overflow = 1;
    }
}

// The light-path steps give each proposal a group of lanes: the lanes split
// the job's partitions, and the group's first lane does the per-proposal work
// (flags, sizes, bids, sums).  A partition is a chain of dependent loads and
// atomics (find the slot, exchange, add, look at the summary: about 2.5 us), so
// when the proposals leave threads idle a group gets more lanes than the
// scoring's gs, up to one per partition (colour classes of n = 1e5, k = 8:
// stage + evaluate + commit 85 -> 35 us); a lane count set by the caller stays.
__device__ __forceinline__ int proposal_lanes(const SweepArgs& a, long long np)
{
    int gs = a.gs;
    if (a.gs_set) return gs;
    const long long threads = (long long)gridDim.x * blockDim.x;
    while (gs < 32 && gs < a.kmax && 2 * gs * np <= threads) gs <<= 1;
    return gs;
}

#define PROPOSAL_LOOP(np)                                                                                  \
    const int gs = proposal_lanes(a, np), per = 32 / gs;                                                  \
    const int lane = threadIdx.x & 31, l = lane & (gs - 1);                                               \
    const long long warp0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;                      \
    const long long nwarp = ((long long)gridDim.x * blockDim.x) >> 5;                                     \
    for (long long b0 = warp0 * per; b0 < (np); b0 += nwarp * per)

// Slots of two keys (-1: absent), their first probes in flight together.
__device__ __forceinline__ void table_find_pair(const Slot* t, unsigned long long mask, unsigned long long ka,
                                                unsigned long long kb, long long& sa, long long& sb)
{
    const unsigned long long ha = hash_key(ka) & mask, hb = hash_key(kb) & mask;
    const unsigned long long a = *reinterpret_cast<const volatile unsigned long long*>(&t[ha].key);
    const unsigned long long b = *reinterpret_cast<const volatile unsigned long long*>(&t[hb].key);
    sa = a == ka ? (long long)ha : a == kEmpty ? -1 : table_find(t, mask, ka);
    sb = b == kb ? (long long)hb : b == kEmpty ? -1 : table_find(t, mask, kb);
}

__device__ __forceinline__ long long group_sum64(long long x, int gs)
{
    for (int o = gs >> 1; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
    return x;
}

// Singleton guard, and staged deltas of the kept proposals.  Staging never
// fails: if the table runs short of slots the sweep is abandoned
// (st->overflow) before anything is committed, and the sweep end schedules a
// larger table and a retry.
__device__ __forceinline__ void stage_phase(const SweepArgs& a)
{
    extern __shared__ long long dyn_jobs[];
    DevState* st = a.st;
    if (st->skip || st->err || st->heavy) return;
    JobAcc acc(job_smem_init(a.jobs, dyn_jobs), reinterpret_cast<long long*>(&a.js[0].np1), kJobStride);
    const unsigned long long mask = st->mask;
    const long long np = (long long)st->nprop;
    PROPOSAL_LOOP(np)
    {
        const long long p = b0 + lane / gs;
        int job = -1, ins_count = 0;
        if (p < np) {
            const int v = a.pv[p], ca = a.pa[p], cb = a.pb[p];
            const bool keep = !(a.size[ca] == 1 && a.size[cb] == 1) || cb < ca;
            if (l == 0) a.pflag[p] = keep ? 1 : 0;
            if (keep) {
                const int j = a.jid[v];
                const JobInfo& J = a.job[j];
                if (l == 0) {
                    job = j;
                    atomicAdd(&a.dsize[ca], -1);
                    atomicAdd(&a.dsize[cb], 1);
                }
                const int* gv = a.G + row_of(J, v);
                for (int i = l; i < J.k; i += gs) {
                    const int g = gv[i];
                    bool ins = false;
                    long long sa, sb;
                    table_find_pair(a.table, mask, ckey(ca, g), ckey(cb, g), sa, sb);
                    if (sb < 0) sb = table_find_or_insert(a.table, mask, ckey(cb, g), &ins);
                    ins_count += ins;
                    if (sa < 0) {
                        set_err(st, CC_ERR_INVALID);  // the vertex's own key must exist
                    } else if (sb < 0) {
                        st->overflow = 1;
                    } else {
                        atomicAdd(&a.table[sa].dlt, -1);
                        atomicAdd(&a.table[sb].dlt, 1);
                    }
                }
            }
        }
        count_inserts(st, ins_count, mask);
        if (job >= 0) acc.add(job, 1);
    }
    job_acc_finish(acc, a.jobs);
}

// dF(P1) per job = k sum_c ((s+ds)^2 - s^2) - 2 sum_keys ((n+dn)^2 - n^2),
// written as a sum over the staged contributions: each +-1 added to an entry
// x with final delta d_x contributes +-(2 x + d_x).
__device__ __forceinline__ void eval_phase(const SweepArgs& a)
{
    extern __shared__ long long dyn_jobs[];
    DevState* st = a.st;
    if (st->skip || st->err || st->overflow || st->heavy) return;
    JobAcc acc(job_smem_init(a.jobs, dyn_jobs), &a.js[0].dF, kJobStride);
    const unsigned long long mask = st->mask;
    const long long np = (long long)st->nprop;
    PROPOSAL_LOOP(np)
    {
        const long long p = b0 + lane / gs;
        long long keys = 0, sizes = 0;
        int job = -1;
        if (p < np && a.pflag[p]) {
            const int v = a.pv[p], ca = a.pa[p], cb = a.pb[p];
            const int j = a.jid[v];
            const JobInfo& J = a.job[j];
            const int* gv = a.G + row_of(J, v);
            for (int i = l; i < J.k; i += gs) {
                const int g = gv[i];
                long long sa, sb;
                table_find_pair(a.table, mask, ckey(ca, g), ckey(cb, g), sa, sb);
                if (sa < 0 || sb < 0) {
                    set_err(st, CC_ERR_INVALID);  // staged keys must exist
                    continue;
                }
                const Slot* A = a.table + sa;
                const Slot* B = a.table + sb;
                const int na = A->cnt, da = A->dlt, nb = B->cnt, db = B->dlt;
                keys += -(2LL * na + da) + (2LL * nb + db);
            }
            if (l == 0) {
                job = j;
                sizes = (long long)J.k * (-(2LL * a.size[ca] + a.dsize[ca]) + (2LL * a.size[cb] + a.dsize[cb]));
            }
        }
        keys = group_sum64(keys, gs);
        if (job >= 0) acc.add(job, -2 * keys + sizes);
    }
    job_acc_finish(acc, a.jobs);
}

__device__ __forceinline__ void decide_phase(const SweepArgs& a, int t0, int stride)
{
    DevState* st = a.st;
    if (st->skip || st->heavy) return;
    for (int j = t0; j < a.jobs; j += stride) {
        JobState& s = a.js[j];
        if (s.stop) continue;
        if (st->err || st->overflow) {
            s.mode = 0;
            continue;
        }
        if (s.np1 > 0 && s.dF < 0) {
            s.mode = 1;
            s.dF_p1 = s.dF;
            s.moves = s.np1;
        } else if (s.nprop > 0) {
            s.mode = 2;
            st->match = 1;
            s.dF_p1 = s.np1 > 0 ? s.dF : 0;
            s.dF = 0;
            s.moves = 0;
        } else {
            s.mode = 0;
            s.dF = 0;
        }
    }
}

// Proposals of a job that falls back to the matching (mode 2): undo their
// staged deltas (light sweeps) and bid (dD, v) at both clusters.
__device__ __forceinline__ void bid_phase(const SweepArgs& a)
{
    DevState* st = a.st;
    if (st->skip || st->err) return;
    const bool staged = !st->heavy;
    const unsigned long long mask = st->mask;
    const long long np = (long long)st->nprop;
    PROPOSAL_LOOP(np)
    {
        const long long p = b0 + lane / gs;
        if (p >= np) continue;
        const int v = a.pv[p], ca = a.pa[p], cb = a.pb[p];
        const int j = a.jid[v];
        if (a.js[j].mode != 2) continue;
        if (staged && a.pflag[p]) {
            const JobInfo& J = a.job[j];
            const int* gv = a.G + row_of(J, v);
            for (int i = l; i < J.k; i += gs) {
                const int g = gv[i];
                const long long sa = table_find(a.table, mask, ckey(ca, g));
                const long long sb = table_find(a.table, mask, ckey(cb, g));
                if (sa >= 0) a.table[sa].dlt = 0;
                if (sb >= 0) a.table[sb].dlt = 0;
            }
            if (l == 0) {
                a.dsize[ca] = 0;
                a.dsize[cb] = 0;
            }
        }
        if (l == 0) {
            const unsigned long long key = pack_key(a.pg[p], v);
            atomicMin(&a.best[ca], key);
            atomicMin(&a.best[cb], key);
        }
    }
}

// Fallback: a proposal is committed iff its (dD, v) is the least at both of
// its clusters; the committed moves touch pairwise-disjoint clusters, so
// their objective changes add exactly.  This pass marks the winners and
// inserts their target keys.  It runs before any count of any job changes,
// so that a table overflow abandons the whole sweep with nothing committed.
__device__ __forceinline__ void match_keys_phase(const SweepArgs& a)
{
    DevState* st = a.st;
    if (st->skip || st->err) return;
    const unsigned long long mask = st->mask;
    const long long np = (long long)st->nprop;
    PROPOSAL_LOOP(np)
    {
        const long long p = b0 + lane / gs;
        int ins_count = 0;
        if (p < np) {
            const int v = a.pv[p], ca = a.pa[p], cb = a.pb[p];
            const int j = a.jid[v];
            const unsigned long long key = pack_key(a.pg[p], v);
            if (a.js[j].mode == 2 && a.best[ca] == key && a.best[cb] == key) {
                if (l == 0) a.pflag[p] = 2;
                const JobInfo& J = a.job[j];
                const int* gv = a.G + row_of(J, v);
                for (int i = l; i < J.k; i += gs) {
                    bool ins = false;
                    if (table_find_or_insert(a.table, mask, ckey(cb, gv[i]), &ins) < 0) st->overflow = 1;
                    ins_count += ins;
                }
            }
        }
        count_inserts(st, ins_count, mask);
    }
}

// The light commit of P1 (mode 1: C, the staged size and count deltas folded
// in) or the move of a matching winner (mode 2).  Skipped entirely after an
// overflow.
__device__ __forceinline__ void commit_phase(const SweepArgs& a)
{
    extern __shared__ long long dyn_jobs[];
    DevState* st = a.st;
    if (st->skip || st->err || st->overflow) return;
    long long* sh = job_smem_init(2 * a.jobs <= kSmemJobs ? a.jobs : 0, dyn_jobs);
    if (sh) {
        for (int j = threadIdx.x; j < a.jobs; j += blockDim.x) sh[a.jobs + j] = 0;
        __syncthreads();
    }
    JobAcc mv(sh, reinterpret_cast<long long*>(&a.js[0].moves), kJobStride);
    JobAcc df(sh ? sh + a.jobs : nullptr, &a.js[0].dF, kJobStride);
    const unsigned long long mask = st->mask;
    const long long np = (long long)st->nprop;
    PROPOSAL_LOOP(np)
    {
        const long long p = b0 + lane / gs;
        long long live = 0, dF = 0, moved = 0;
        int job = -1;
        if (p < np) {
            const int v = a.pv[p], ca = a.pa[p], cb = a.pb[p];
            const int j = a.jid[v];
            const int mode = a.js[j].mode;
            const JobInfo& J = a.job[j];
            const int* gv = a.G + row_of(J, v);
            if (mode == 1 && a.pflag[p]) {
                if (l == 0) {
                    a.C[v] = cb;
                    a.chg[ca] = st->stamp;
                    a.chg[cb] = st->stamp;
                    int d = atomicExch(&a.dsize[ca], 0);
                    if (d) atomicAdd(&a.size[ca], d);
                    d = atomicExch(&a.dsize[cb], 0);
                    if (d) atomicAdd(&a.size[cb], d);
                }
                for (int i = l; i < J.k; i += gs) {
                    const int g = gv[i];
                    long long sa, sb;
                    table_find_pair(a.table, mask, ckey(ca, g), ckey(cb, g), sa, sb);
                    if (sa < 0 || sb < 0) {
                        set_err(st, CC_ERR_INVALID);
                        continue;
                    }
                    // both sides' atomics in flight together
                    const int da = atomicExch(&a.table[sa].dlt, 0), db = atomicExch(&a.table[sb].dlt, 0);
                    const int oa = da ? atomicAdd(&a.table[sa].cnt, da) : 1;
                    const int ob = db ? atomicAdd(&a.table[sb].cnt, db) : 1;
                    if (da) live += (oa == 0) - (oa + da == 0);
                    if (db) live += (ob == 0) - (ob + db == 0);
                    if (da) summ_update(a, J, ca, i, g, da);
                    if (db) summ_update(a, J, cb, i, g, db);
                }
            } else if (mode == 2 && a.pflag[p] == 2) {
                if (l == 0) {
                    job = j;
                    a.C[v] = cb;
                    a.chg[ca] = st->stamp;
                    a.chg[cb] = st->stamp;
                    atomicAdd(&a.size[ca], -1);
                    atomicAdd(&a.size[cb], 1);
                    moved = 1;
                    dF = 2LL * a.pg[p];
                }
                for (int i = l; i < J.k; i += gs) {
                    const int g = gv[i];
                    long long sa, sb;
                    table_find_pair(a.table, mask, ckey(ca, g), ckey(cb, g), sa, sb);
                    if (sa < 0 || sb < 0) {
                        set_err(st, CC_ERR_INVALID);
                        continue;
                    }
                    const int oa = atomicAdd(&a.table[sa].cnt, -1);
                    const int ob = atomicAdd(&a.table[sb].cnt, 1);
                    live += (ob == 0) - (oa == 1);
                    summ_update(a, J, ca, i, g, -1);
                    summ_update(a, J, cb, i, g, 1);
                }
            }
        }
        warp_add64(live, &st->live);
        if (job >= 0) {
            mv.add(job, moved);
            df.add(job, dF);
        }
    }
    job_acc_finish(mv, a.jobs);
    job_acc_finish(df, a.jobs);
}

__device__ __forceinline__ void match_reset_phase(const SweepArgs& a)
{
    DevState* st = a.st;
    if (st->skip) return;
    const long long np = (long long)st->nprop;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < np; p += stride) {
        if (a.js[a.jid[a.pv[p]]].mode != 2) continue;
        a.best[a.pa[p]] = kEmpty;
        a.best[a.pb[p]] = kEmpty;
    }
}

// Per job: objective, history record, stop.  An abandoned sweep changes no job.
__device__ __forceinline__ void end_jobs_phase(const SweepArgs& a, int t0, int stride)
{
    DevState* st = a.st;
    if (st->skip || st->err || st->overflow) return;
    for (int j = t0; j < a.jobs; j += stride) {
        JobState& s = a.js[j];
        if (s.stop) continue;
        if (s.mode != 0) s.F += s.dF;
        cc_sweep_info r;
        r.proposals = (int64_t)s.nprop;
        r.p1 = (int64_t)s.np1;
        r.dF_p1 = s.dF_p1;
        r.fallback = s.mode == 2 ? 1 : 0;
        r.moves = (int64_t)s.moves;
        r.F = s.F;
        if (a.colour_mode) {
            // a colour class: add it to the sweep's totals; the sweep ends
            // with its last class
            s.t_prop += r.proposals;
            s.t_p1 += r.p1;
            s.t_dFp1 += r.dF_p1;
            s.t_fb += r.fallback;
            s.t_moves += r.moves;
            if (st->cls + 1 < st->ncls) continue;
            r.proposals = s.t_prop;
            r.p1 = s.t_p1;
            r.dF_p1 = s.t_dFp1;
            r.fallback = s.t_fb;
            r.moves = s.t_moves;
            s.t_prop = s.t_p1 = s.t_dFp1 = s.t_fb = s.t_moves = 0;
        }
        if (s.sweeps < a.hist_cap) a.hist[(long long)j * a.hist_cap + s.sweeps] = r;
        s.sweeps += 1;
        s.run_sweeps += 1;
        if (r.proposals == 0 || s.run_sweeps >= st->run_limit) s.stop = 1;
        else atomicAdd(&st->active, 1);
    }
}

__device__ __forceinline__ void end_phase(const SweepArgs& a)
{
    DevState* st = a.st;
    if (st->skip) return;
    st->run_bodies += 1;
    if (st->err) {
        st->stop = 1;
        return;
    }
    const unsigned long long cap = st->mask + 1;
    st->build_small = 0;  // a rebuild at the end of a sweep holds every key
    if (st->overflow) {
        // nothing was committed: retry this sweep after rebuilding into twice
        // the capacity (the staged deltas are discarded with the old table).
        // A heavy sweep sizes its table for every key it can create, so it
        // cannot overflow; if it did, jobs that kept P1 have moved already
        // and a retry would be wrong, so that is reported instead.
        if (cap >= a.mask_max + 1 || st->heavy) {
            set_err(st, CC_ERR_TABLE_FULL);
            st->stop = 1;
            return;
        }
        st->new_mask = 2 * cap - 1;
        st->abort = 1;
        st->rebuild = 1;
        st->retries += 1;
        st->stamp -= 1;  // the retry is the same sweep: it reuses the stamp
        return;
    }
    st->all_active = 0;
    if (a.colour_mode && st->cls + 1 < st->ncls) {
        st->cls += 1;  // the sweep goes on with the next colour class
        st->stop = 0;
    } else {
        st->cls = 0;
        st->stop = st->active == 0 ? 1 : 0;
    }
    // compaction: rebuild without the dead keys when occupied slots pass one
    // half of the capacity; the new capacity holds the live keys plus k x
    // (proposals of this sweep), a forecast of the next sweep's new keys, at
    // load <= 1/2.  (Summary rows settle most of each score, so a table larger
    // than needed costs little; it is not shrunk otherwise.)
    const unsigned long long live = (unsigned long long)st->live;
    const unsigned long long want = 2 * (live + st->pkeys);
    unsigned long long c = a.cap_min;
    while (c < want && c < a.mask_max + 1) c <<= 1;
    if (st->tvalid && !st->small && st->used > cap / 2) {
        st->new_mask = c - 1;
        st->rebuild = 1;
    } else {
        st->rebuild = 0;
    }
}

}  // namespace

}  // namespace ccg

// Device code of the table rebuild (see setup.cu for the kernels that run it
// one step at a time, persist.cu for the run kernel that calls the steps
// between its grid barriers).  Every function is one step over the whole
// grid: blocks take their share by blockIdx and gridDim.
#pragma once

#include "cc_internal.cuh"

namespace ccg {

namespace {

// ---- table rebuild ------------------------------------------------------
// The table is rebuilt from C alone: list the vertices cluster by cluster
// (counting sort: an exclusive scan of the sizes gives each cluster's first
// position), clear the capacity being built, then insert the keys with
// partitions innermost per member, so that the 32 lanes of a warp hold
// consecutive members of (mostly) one cluster for one partition: equal keys
// are merged with __match_any_sync and added with one atomic.  The summary
// rows follow from the rebuilt counts.  All steps are skipped unless a
// rebuild is pending (conditional) and run unconditionally otherwise.
//
// A heavy sweep whose P1 leaves many label rows in clusters of at most kSmall
// members (the first sweep of a run, above all) builds a partial table: those
// clusters get neither keys nor summary rows, since the next sweep's scoring
// compares v's label row with their few members' rows instead (the member
// list is part of the rebuild), and a sweep that finds a partial table is
// heavy, so nothing else looks for their keys.  On the kNN workload (n = 2e6,
// k = 50) 99.5% of the vertices are in such clusters after sweep 1, and its
// rebuild shrank from 62.5M keys in 2^28 slots (5.8 ms) to 0.2M keys.  Not
// worth it below a quarter of the rows: the full table then costs little and
// lets a light sweep follow.

__device__ __forceinline__ bool rebuild_off(const DevState* st, int conditional)
{
    return conditional && (!st->rebuild || st->err);
}

// Whether the rebuild's sizes are still to be looked over (see size_build).
__device__ __forceinline__ bool to_size(const DevState* st, int conditional)
{
    return conditional && st->heavy && !st->rollback && !st->sized;
}

// Label rows of cluster c (sz members) that a partial table would leave out.
__device__ __forceinline__ unsigned long long small_rows(const SweepArgs& a, long long c, int sz)
{
    return sz >= 1 && sz <= kSmall ? (unsigned long long)sz * a.job[a.jid[c]].k : 0ull;
}

__device__ __forceinline__ void add_small_rows(DevState* st, unsigned long long x)
{
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if ((threadIdx.x & 31) == 0 && x) atomicAdd(&st->small_keys, x);
}

// One thread, once the sizes after P1 are known: partial or full table, and
// its capacity.  First a tight one: the occupied slots of the sweep start
// (the moves of a heavy sweep mostly merge keys) at load <= 1/2, with room
// below the fill limit for the new keys of a light sweep that may follow a
// full table (2 x sum k n / 8 at most).  After a partial table the keys of
// the small clusters were not counted; the sweep that merges them leaves
// 11-13% of their rows as keys on the kNN and LFR-style workloads, and a
// quarter is assumed; but three quarters of the rows that are still in small
// clusters, whose members need not agree on much (jobs with noisy labels that
// end with such clusters: a light sweep follows, so the table is full).  The build checks that the keys fit (build_check) and
// otherwise builds again at the capacity that holds every key.
__device__ __forceinline__ void size_build(const SweepArgs& a)
{
    DevState* st = a.st;
    st->sized = 1;
    const unsigned long long total = a.keys;
    const bool partial = !st->build_light && 4 * st->small_keys >= total;
    unsigned long long c = st->safe_mask + 1;
    unsigned long long est = !st->tvalid ? total : st->small ? st->used + (st->keys_all - st->used) / 4 : st->used;
    unsigned long long room = 2 * ((total + 7) / 8);
    if (partial) {
        const unsigned long long rest = total - st->small_keys;
        unsigned long long p = a.cap_min;
        while (p < 2 * rest && p < c) p <<= 1;
        c = p;
        if (est > rest) est = rest;
        room = 0;
    } else if (st->small && est < st->small_keys / 4 * 3) {
        est = st->small_keys / 4 * 3;
    }
    unsigned long long t = a.cap_min;
    while ((t < 2 * est || t - (t >> 3) < est + room) && t < c) t <<= 1;
    st->build_small = partial ? kSmall : 0;
    st->retry_mask = c - 1;
    st->tight = (t < c && a.tight_mode != 1) ? 1 : 0;
    st->new_mask = (st->tight ? t : c) - 1;
}

// Clears the slots of the capacity being built (st->new_mask + 1 of them),
// the summary rows, the occupied-slot counter, and the staged size deltas
// after an abandoned sweep.  Summary rows: those of the live clusters that
// the table holds (a warp per 32 cluster ids, the lanes across each live
// row), which are the rows the rebuild fills and the sweeps read.  The row of
// a dead cluster is never read again, since no move enters an empty cluster,
// except with empty_moves (a vertex may found a cluster under its own,
// possibly dead, id); then every row of a full table is cleared.
__device__ __forceinline__ void table_clear_phase(const SweepArgs& a, long long rows, int conditional)
{
    DevState* st = a.st;
    if (rebuild_off(st, conditional)) return;
    const unsigned long long cap = st->new_mask + 1;
    const int small = conditional ? st->build_small : 0;
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    const unsigned long long t0 = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
    for (unsigned long long s = t0; s < cap; s += stride)
        reinterpret_cast<ulonglong2*>(a.table)[s] = make_ulonglong2(kEmpty, 0ull);
    const int4 none = make_int4(-1, 0, -1, 0);
    if (a.empty_moves && !small) {
        for (unsigned long long r = t0; r < (unsigned long long)rows; r += stride) a.summ[r] = none;
    } else {
        const int lane = threadIdx.x & 31;
        for (unsigned long long x0 = t0 - lane; x0 < (unsigned long long)a.n; x0 += stride) {
            const unsigned long long x = x0 + lane;
            unsigned live = __ballot_sync(0xffffffffu, x < (unsigned long long)a.n && a.size[x] > small);
            while (live) {
                const long long xx = (long long)x0 + __ffs(live) - 1;
                live &= live - 1;
                const JobInfo& J = a.job[a.jid[xx]];
                int4* row = a.summ + row_of(J, xx);
                for (int q = lane; q < J.kp; q += 32) row[q] = none;
            }
        }
    }
    if (st->abort)
        for (unsigned long long v = t0; v < (unsigned long long)a.n; v += stride) a.dsize[v] = 0;
    if (t0 == 0) st->used = 0;
}

__device__ __forceinline__ int warp_incl_scan(int x, int lane)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    return x;
}

// Cluster ids of a tile of vertices counted in shared memory, so that a block
// adds to a cluster's word in global memory once per tile instead of once per
// vertex: adds to one word take about 10 ns each, and the largest clusters
// hold several percent of the vertices (n = 1e6, 200 clusters: 233 -> 45 us).
// A tile is four vertices per thread, or one up to kSmallTiles vertices, where
// the time is a block's chain of steps (n = 3000: scatter 4.6 -> 2.6 us; n =
// 100,003 6.4 -> 3.6).
constexpr int kTile = 4 * kBlock;
constexpr long long kSmallTiles = 1 << 17;
struct TileCount {
    int key[2 * kTile], cnt[2 * kTile];
};

// All threads of the block; ids: this thread's kPer (-1: none).  Leaves the
// entry of each in slot and its number among the tile's equal ones in rank.
template <int kPer>
__device__ __forceinline__ void tile_count(TileCount* tc, const int (&id)[kPer], int (&slot)[kPer], int (&rank)[kPer])
{
    constexpr int kEntries = 2 * kPer * kBlock;
    for (int s = threadIdx.x; s < kEntries; s += kBlock) {
        tc->key[s] = -1;
        tc->cnt[s] = 0;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
        slot[q] = rank[q] = 0;
        if (id[q] < 0) continue;
        int h = (int)(((unsigned)id[q] * 0x9E3779B1u) >> 16) & (kEntries - 1);
        // half as many ids as entries at most: an empty one is found
        for (int p = 0; p < kEntries; ++p) {
            const int old = atomicCAS(&tc->key[h], -1, id[q]);
            if (old == -1 || old == id[q]) break;
            h = (h + 1) & (kEntries - 1);
        }
        slot[q] = h;
        rank[q] = atomicAdd(&tc->cnt[h], 1);
    }
    __syncthreads();
}

template <int kPer>
__device__ __forceinline__ void scatter_tiles(const SweepArgs& a, bool undone, TileCount* tc)
{
    constexpr int kThis = kPer * kBlock;
    for (long long t0 = (long long)blockIdx.x * kThis; t0 < a.n; t0 += (long long)gridDim.x * kThis) {
        int id[kPer], slot[kPer], rank[kPer];
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            const long long v = t0 + q * kBlock + threadIdx.x;
            id[q] = v < a.n ? a.C[v] : -1;
        }
        tile_count(tc, id, slot, rank);
        for (int s = threadIdx.x; s < 2 * kThis; s += kBlock)
            if (tc->cnt[s]) tc->cnt[s] = atomicAdd(&a.cursor[tc->key[s]], tc->cnt[s]);
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            const long long v = t0 + q * kBlock + threadIdx.x;
            if (id[q] < 0) continue;
            const int pos = tc->cnt[slot[q]] + rank[q];
            if (pos < a.n) a.members[pos] = (int)v;
            else set_err(a.st, CC_ERR_INVALID);  // sizes inconsistent with C
            // P1 is being undone: what h_eval computed under it no longer holds
            if (undone && a.chg[id[q]] == a.st->stamp) a.own[v].y = kOwnNever;
        }
        __syncthreads();
    }
}

__device__ __forceinline__ void members_scatter_phase(const SweepArgs& a, int conditional, TileCount* tc)
{
    if (rebuild_off(a.st, conditional)) return;
    const bool undone = conditional && a.st->rollback;
    if (a.n <= kSmallTiles) scatter_tiles<1>(a, undone, tc);
    else scatter_tiles<4>(a, undone, tc);
}

// Largest 64-bit value over the lanes of a contiguous lane segment [lane,
// end) of the warp, left in the segment's first lane (every lane must call it).
__device__ __forceinline__ unsigned long long segment_max(unsigned long long x, int lane, int end)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_down_sync(0xffffffffu, x, o);
        if (lane + o < end && y > x) x = y;
    }
    return x;
}

// Inserts the keys of every member of a cluster the table holds (partitions
// innermost, equal keys of a warp merged with __match_any_sync and added
// once).  Members are listed cluster by cluster, so a cluster whose members
// all lie in one warp's 32 entries gets its exact counts inside that warp:
// the warp then writes the cluster's summary entries itself (the two most
// frequent labels, ties to the larger id, as the table scan would rank them)
// and marks those keys so that the scan skips them.  Keys of clusters spread
// over several warps are left to the scan.
// A tight attempt (see build_check) gives every insert kTightProbes probes;
// an insert that finds no slot within them flags the attempt as failed, and
// the warps stop inserting.  At load 1/2 the longest chain of n keys is about
// ln n / 0.19 slots (79 for 2^22, 97 for 2^27), so 128 do not fail an attempt
// that fits; and a warp looks at the flag every 16 probes, for in a table that
// overflows every chain is long (2500 jobs of n = 100 with random labels, whose
// clusters merge fewer keys than size_build assumes: the failed attempt took 484
// of 875 us of its sweep with 256 probes and no look, 128 so).
constexpr unsigned kTightProbes = 128, kLookProbes = 16;

// Claims an empty slot for key if on; returns the key found there (key itself
// where off).  One predicated instruction, so that several follow each other
// without waiting for a result.
__device__ __forceinline__ unsigned long long key_cas_if(unsigned on, unsigned long long* slot, unsigned long long key)
{
    unsigned long long old = key;
    asm volatile(
        "{\n\t"
        ".reg .pred p;\n\t"
        "setp.ne.u32 p, %3, 0;\n\t"
        "@p atom.relaxed.gpu.global.cas.b64 %0, [%1], %4, %2;\n\t"
        "}"
        : "+l"(old)
        : "l"(slot), "l"(key), "r"(on), "l"(kEmpty)
        : "memory");
    return old;
}

__device__ __forceinline__ void table_build_phase(const SweepArgs& a, int conditional)
{
    DevState* st = a.st;
    if (rebuild_off(st, conditional)) return;
    __shared__ unsigned long long s_used;
    if (threadIdx.x == 0) s_used = 0;
    // tight attempts are made only by the heavy sweep's rebuild inside a
    // sweep graph; a rebuild the host asks for is never one
    const bool tight = conditional && st->tight != 0;
    const int small = conditional ? st->build_small : 0;
    const unsigned long long mask = st->new_mask;
    const unsigned first_stop = tight ? kLookProbes : ~0u;  // probes of a key before the first look at the limits
    const int lane = threadIdx.x & 31;
    unsigned created = 0;  // slots this lane created
    // an item is a window of 32 members and a run of quads of partitions: a
    // window alone is too long a chain (one round of inserts per quad) for
    // the warps to end together when they get only a few each
    const long long nwarps = (long long)gridDim.x * kWarpsPerBlock, windows = (a.n + 31) >> 5;
    const int kq = (a.kmax + 3) >> 2;
    const int parts = (int)max(1LL, min((long long)kq, (8 * nwarps + windows - 1) / windows));
    const int run_q = (kq + parts - 1) / parts;
    __shared__ int s_taken;
    const WarpQueue queue{&s_taken};
    queue.start();
    for (long long item = queue.next(); item < windows * parts; item = queue.next()) {
        if (tight && __any_sync(0xffffffffu, *reinterpret_cast<volatile int*>(&st->build_fail) != 0)) break;
        const long long window = item / parts;
        const int first_i = 4 * run_q * (int)(item - window * parts), last_i = min(a.kmax, first_i + 4 * run_q);
        const long long wb = window * 32, m = wb + lane;  // the warp's members
        bool valid = m < a.n;
        int v = 0, c = 0, k = 0, seg_end = lane + 1;
        bool whole = false;
        const int* row = a.G;
        int4* S = a.summ;
        if (valid) {
            v = a.members[m];
            c = a.C[v];
            if (a.size[c] <= small) valid = false;
        }
        if (!__any_sync(0xffffffffu, valid)) continue;
        if (valid) {
            const JobInfo& J = a.job[a.jid[v]];
            k = J.k;
            if (k <= first_i) valid = false;
        }
        if (!__any_sync(0xffffffffu, valid)) continue;
        if (valid) {
            const JobInfo& J = a.job[a.jid[v]];
            row = a.G + row_of(J, v);
            // after the scatter, cursor[c] is one past the cluster's last member
            const long long end = a.cursor[c], first = end - a.size[c];
            whole = first >= wb && end <= wb + 32;
            if (whole) seg_end = (int)(end - wb);
            S = a.summ + row_of(J, c);
        }
        const int hl = whole ? (int)((long long)a.cursor[c] - a.size[c] - wb) : lane;  // the cluster's first lane
        const bool head = whole && hl == lane;
        // the warp's whole clusters need the summary maxima; a warp without
        // any skips them
        const bool any_whole = __any_sync(0xffffffffu, whole);
        const int4* G4 = reinterpret_cast<const int4*>(row);
        // lanes holding members of this lane's cluster (a contiguous run)
        const int cl = valid ? c : -1 - lane;
        const int up = __shfl_up_sync(0xffffffffu, cl, 1);
        const unsigned heads = __ballot_sync(0xffffffffu, lane == 0 || up != cl);
        const int run0 = 31 - __clz(heads & (0xffffffffu >> (31 - lane)));
        const unsigned above = lane == 31 ? 0u : heads & (0xfffffffeu << lane);
        const unsigned run = (0xffffffffu << run0) & (above ? (1u << (__ffs(above) - 1)) - 1u : 0xffffffffu);
        // a whole cluster's new slots are marked (their summary entry is final;
        // the scan clears the mark before any sweep stages deltas); such a
        // key is added once
        const unsigned long long mark = whole ? (1ull << 32) : 0ull;
        // four partitions at a time: one quad of the label row, and the four
        // keys' first CASes issued before any result is used
        for (int i0 = first_i; i0 < last_i; i0 += 4) {
            int4 g4 = make_int4(0, 0, 0, 0);
            if (valid && i0 < k) g4 = __ldg(G4 + (i0 >> 2));
            const int gq[4] = {g4.x, g4.y, g4.z, g4.w};
            // only the labels, the counts (a byte each) and the leader bits
            // stay live; keys and slots are computed again for each probe
            unsigned cnts = 0, pend = 0;
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const bool on = valid && i0 + b < k;
                const unsigned same = __match_any_sync(0xffffffffu, on ? gq[b] : -1) & run;
                cnts |= (unsigned)__popc(same) << (8 * b);
                pend |= (on && (__ffs(same) - 1) == lane) ? 1u << b : 0u;
            }
            // probe round p: the p-th slot of every key not placed yet, all
            // of them in flight together (a lane's keys collide one by one,
            // but the warp waits only for its longest chain, not for their sum)
            unsigned stop = first_stop > mask ? (unsigned)mask + 1u : first_stop;
            for (unsigned p = 0; pend; ++p) {
                if (p == stop) {
                    if (!tight) {
                        set_err(st, CC_ERR_TABLE_FULL);
                        break;
                    }
                    if (p >= kTightProbes || p > mask) st->build_fail = 1;
                    if (*reinterpret_cast<volatile int*>(&st->build_fail)) break;
                    stop = p + kLookProbes > mask ? (unsigned)mask + 1u : p + kLookProbes;
                }
                unsigned long long old[4];
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    const unsigned long long key = ckey(c, gq[b]);
                    old[b] = key_cas_if(pend >> b & 1u, &a.table[(hash_key(key) + p) & mask].key, key);
                }
#pragma unroll
                for (int b = 0; b < 4; ++b)
                    if (pend >> b & 1u) {
                        const unsigned long long key = ckey(c, gq[b]);
                        if (old[b] != kEmpty && old[b] != key) continue;
                        created += old[b] == kEmpty;
                        // {count, mark}: nothing waits for the sum
                        atomicAdd(reinterpret_cast<unsigned long long*>(&a.table[(hash_key(key) + p) & mask].cnt),
                                  mark | (cnts >> (8 * b) & 255u));
                        pend &= ~(1u << b);
                    }
            }
            if (!any_whole) continue;
            // summary entries of the whole clusters: the two largest (count, label)
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const bool on = valid && i0 + b < k;
                const unsigned long long mine =
                    (whole && on) ? ((unsigned long long)(cnts >> (8 * b) & 255u) << 32) | (unsigned)gq[b] : 0ull;
                const unsigned long long top1 = segment_max(mine, lane, seg_end);
                const unsigned long long t1 = __shfl_sync(0xffffffffu, top1, hl);
                const unsigned long long other = (mine != 0 && (unsigned)mine != (unsigned)t1) ? mine : 0ull;
                const unsigned long long top2 = segment_max(other, lane, seg_end);
                if (head && on) {
                    const int d2 = top2 ? (int)(unsigned)top2 : -1, m2 = (int)(top2 >> 32);
                    S[b * ((k + 3) >> 2) + (i0 >> 2)] = make_int4((int)(unsigned)top1, (int)(top1 >> 32), d2, m2);
                }
            }
        }
    }
    // one add per block: st->used is a single word that every block updates
    for (int o = 16; o > 0; o >>= 1) created += __shfl_xor_sync(0xffffffffu, created, o);
    if (lane == 0 && created) atomicAdd(&s_used, (unsigned long long)created);
    __syncthreads();
    if (threadIdx.x == 0 && s_used) atomicAdd(&st->used, s_used);
}

// Summary rows of the rebuilt table for the keys the build left unmarked
// (clusters spread over several warps).  Each half of a row entry reads as
// one unsigned 64-bit value (count << 32 | label id); every such slot offers
// its (count, label) to the entry, which keeps the two largest by a 16-byte
// compare-and-swap (ties to the larger id; cleared entries hold count 0 and
// label -1, below any real key).  Content does not depend on the order of
// the offers.  Marked slots only get their mark cleared.
__device__ __forceinline__ void summ_top_phase(const SweepArgs& a, int conditional)
{
    DevState* st = a.st;
    if (rebuild_off(st, conditional) || st->again) return;
    const unsigned long long cap = st->new_mask + 1;
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    for (unsigned long long s = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; s < cap; s += stride) {
        const ulonglong2 e = reinterpret_cast<const ulonglong2*>(a.table)[s];
        const int cnt = (int)(unsigned)(e.y & 0xffffffffull);
        if (e.x == kEmpty || cnt <= 0) continue;
        if ((e.y >> 32) != 0) {
            a.table[s].dlt = 0;  // summary done by the build
            continue;
        }
        const int x = (int)(e.x >> 32), g = (int)(unsigned)(e.x & 0xffffffffull);
        const int job = a.jid[x];
        const JobInfo& J = a.job[job];
        int4* E = a.summ + row_of(J, x) + summ_at(J, g >> J.lshift);
        const unsigned long long kn = ((unsigned long long)(unsigned)cnt << 32) | (unsigned)g;
        const volatile unsigned long long* Ev = reinterpret_cast<const volatile unsigned long long*>(E);
        ulonglong2 cur = make_ulonglong2(Ev[0], Ev[1]);
        // lock-free: every failed swap means another offer went in; bounded
        // all the same
        for (int tries = 0; kn > cur.y; ++tries) {
            if (tries >= (1 << 20)) {
                set_err(st, CC_ERR_INVALID);
                break;
            }
            const ulonglong2 nv = kn > cur.x ? make_ulonglong2(kn, cur.x) : make_ulonglong2(cur.x, kn);
            const ulonglong2 old = entry_cas(E, cur, nv);
            if (old.x == cur.x && old.y == cur.y) break;
            cur = old;
        }
    }
}

// Check of a tight attempt, after its build: the table must have taken every
// key within the probe limit, at load <= 1/2, with room left below the fill
// limit for the new keys of a light sweep (at most 2 x sum_j k_j n_j / 8).
// (if it is a full one).  Otherwise the attempt is dropped (the summary pass
// and the done step skip it) and the rebuild runs again at the capacity that
// holds every key it can meet.  One thread.
__device__ __forceinline__ void build_check_phase(const SweepArgs& a, int conditional)
{
    DevState* st = a.st;
    if (threadIdx.x != 0 || rebuild_off(st, conditional)) return;
    int fail = 0;
    if (conditional && st->tight) {
        const unsigned long long cap = st->new_mask + 1, fill = cap - (cap >> 3);
        const unsigned long long room = st->build_small ? 0 : 2 * ((a.keys + 7) / 8);
        fail = st->build_fail || st->used > cap / 2 || st->used + room > fill || a.tight_mode == 2;
    }
    if (fail) st->new_mask = st->retry_mask;
    st->again = fail;
    st->tight = 0;
    st->build_fail = 0;
}

__device__ __forceinline__ void table_done_phase(DevState* st, int conditional)
{
    if (rebuild_off(st, conditional) || st->again) return;
    st->live = (long long)st->used;
    st->mask = st->new_mask;
    st->small = conditional ? st->build_small : 0;
    st->keys_all = st->used + (st->small ? st->small_keys : 0);
    st->rebuild = 0;
    st->abort = 0;
    st->rebuilds += 1;
    st->tvalid = 1;
}

}  // namespace

}  // namespace ccg

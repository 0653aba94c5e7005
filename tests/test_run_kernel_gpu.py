"""The run kernel and the graphs of a run beside the ordinary run: waits that
run out, the autotuned first sweep (against the oracle where there are results;
whole numbers, exact)."""
import ctypes
import os
import subprocess
import sys
import threading
import time

import numpy as np
import pytest

import oracle
from workloads import make_config
from workloads.graphs import csr_from_edges

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SECOND = 10**9


@pytest.fixture(scope="module")
def cc():
    import __graft_entry__

    __graft_entry__.build()
    import paper_2408_11331_gb300 as m

    return m


def _job(n, k, seed=None):
    c = make_config("lfr", n=n, k=k, cmin=10, cmax=300, max_deg=100, seed=n + k if seed is None else seed)
    return c["row_off"], c["col"], c["labels"]


def _options(cc, **fields):
    o = cc.cc_default_options()
    for f, x in fields.items():
        setattr(o, f, x)
    return o


# A limit of 0 makes the first block that waits give up.  The barrier's count
# is then left in the middle of a step; a run after a warm start (or a reset)
# of the same context has to start from a clean one.
@pytest.mark.parametrize("opts", [{}, {"active_set": 1}, {"empty_moves": 1}, {"colour_batched": 1}])
@pytest.mark.parametrize("before", [0, 1, 2])
def test_run_after_a_timeout(cc, opts, before):
    n, k = 6007, 9
    ro, col, lab = _job(n, k)
    run = oracle.colour_run if opts.get("colour_batched") else oracle.sync_run
    kw = {"empty": True} if opts.get("empty_moves") else {}
    ref = run(ro, col, lab, 20, **kw)
    with cc.Consensus(ro, col, lab, _options(cc, **opts)) as job:
        for restart in ("warm", "warm", "reset"):
            for _ in range(before):
                job.sweep()
            job.set_wait_limit(0)
            with pytest.raises(cc.CCError) as e:
                job.run_until_converged(20)
            assert e.value.status == 6
            job.set_wait_limit(SECOND)
            with pytest.raises(cc.CCError):  # the error stays until a restart
                job.run_until_converged(20)
            if restart == "reset":
                job.reset()
            else:
                job.set_cluster_ids(np.arange(n, dtype=np.int32))
            recorded = len(job.history())
            assert job.run_until_converged(20) == ref.sweeps
            assert job.history()[recorded:] == ref.stats
            np.testing.assert_array_equal(job.cluster_ids(), ref.C)
            assert job.objective() == ref.F == job.objective_recompute()


def test_batch_after_a_timeout(cc):
    jobs = [_job(3001, 5), _job(900, 12), _job(40, 3)]
    refs = [oracle.sync_run(*j, 20) for j in jobs]
    with cc.ConsensusBatch(jobs) as batch:
        start = batch.cluster_ids()
        for _ in range(2):
            batch.set_wait_limit(0)
            with pytest.raises(cc.CCError) as e:
                batch.run_until_converged(20)
            assert e.value.status == 6
            batch.set_wait_limit(20 * SECOND)
            batch.set_cluster_ids(start)
            batch.run_until_converged(20)
            np.testing.assert_array_equal(batch.cluster_ids(), np.concatenate([r.C for r in refs]))
            assert [batch.objective(j) for j in range(3)] == [r.F for r in refs]


def test_wait_limit_must_not_be_negative(cc):
    with cc.Consensus(*_job(40, 3)) as job, pytest.raises(cc.CCError):
        job.set_wait_limit(-1)


# The lanes are timed after the first sweep of the first run.  Pairs of vertices
# with the same labels merge in that sweep and the second finds nothing to do,
# so a run that does two sweeps before it times them never times them.  (A
# process of its own: the choices are remembered per process.)
@pytest.mark.parametrize("n", [1000, 40000])
@pytest.mark.parametrize("no_regions", [0, 1])
def test_autotune_after_the_first_sweep(cc, n, no_regions):
    code = f"""
import ctypes, numpy as np, paper_2408_11331_gb300 as cc
def record():
    r = (ctypes.c_int32 * 6)()
    cc._native._check(cc._native.lib.cc_autotune_record(6, r))
    return list(r)
n = {n}
v = np.arange(n)
col = (v ^ 1).astype(np.int32)
lab = np.tile((v // 2).astype(np.int32), (10, 1))
o = cc.cc_default_options()
o.autotune, o.no_regions = 1, {no_regions}
assert not any(record())
with cc.Consensus(np.arange(n + 1, dtype=np.int64), col, lab, o) as job:
    assert job.run_until_converged(20) == 2
    assert np.array_equal(job.cluster_ids(), v // 2 * 2)
    assert len(job.last_run_timing()[0]) == 2
assert record()[0] > 0, record()
"""
    subprocess.run([sys.executable, "-c", code], check=True, cwd=ROOT, timeout=120)


# The caller's own kernels on another stream run beside a run, not after it.
def test_other_streams_run_beside_a_run(cc):
    torch = pytest.importorskip("torch")
    job = cc.Consensus(*_job(200003, 24))
    job.run_until_converged(20)
    started = time.perf_counter()
    job.reset()
    job.run_until_converged(20)
    run_s = time.perf_counter() - started
    stop = threading.Event()

    def runs():
        while not stop.is_set():
            job.reset()
            job.run_until_converged(20)

    other, x = torch.cuda.Stream(), torch.zeros(64, device="cuda")
    with torch.cuda.stream(other):
        x.add_(1)
    torch.cuda.synchronize()
    thread = threading.Thread(target=runs)
    thread.start()
    waits = []
    try:
        for _ in range(100):
            t0 = time.perf_counter()
            with torch.cuda.stream(other):
                x.add_(1)
            other.synchronize()
            waits.append(time.perf_counter() - t0)
            time.sleep(run_s / 3)
    finally:
        stop.set()
        thread.join()
        job.close()
    # half a run on average where it waits for the end of the run
    assert np.median(waits) < run_s / 6, (np.median(waits), run_s)


# Contexts that run at the same time share the GPU, so the number of blocks of a
# launch depends on the others in flight; the results do not.
def test_runs_in_threads(cc):
    sizes = [(1500, 12), (6007, 9), (20011, 12), (3001, 33), (60001, 8), (6007, 20), (900, 40), (20011, 4), (40, 3)]
    jobs = [_job(n, k) for n, k in sizes]
    refs = [oracle.sync_run(*j, 20) for j in jobs]
    wrong = []

    def work(i):
        with cc.Consensus(*jobs[i]) as job:
            for _ in range(12):
                job.reset()
                sweeps = job.run_until_converged(20)
                if (sweeps, job.history()) != (refs[i].sweeps, refs[i].stats) or not np.array_equal(job.cluster_ids(), refs[i].C):
                    wrong.append(i)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong


# Two contexts that each fill the GPU alone: run together they take less than
# one after the other.
def test_two_runs_overlap(cc):
    jobs = [cc.Consensus(*_job(20011, 12, seed)) for seed in (1, 2, 3, 4)]

    def work(job):
        for _ in range(30):
            job.reset()
            job.run_until_converged(20)

    def wall(groups):
        threads = [threading.Thread(target=lambda g=g: [work(j) for j in g]) for g in groups]
        t0 = time.perf_counter()
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        return time.perf_counter() - t0

    wall([jobs])
    alone = min(wall([jobs]) for _ in range(3))
    together = min(wall([[j] for j in jobs]) for _ in range(3))
    for j in jobs:
        j.close()
    assert together < 0.75 * alone, (together, alone)  # one after the other: 0.9


class _Part:
    """A stream on some of the device's SMs (a green context)."""

    def __init__(self, sms):
        self.lib = ctypes.CDLL("libcuda.so.1")
        self.stream, self.green = ctypes.c_void_p(), ctypes.c_void_p()
        dev, count, desc = ctypes.c_int(), ctypes.c_uint(1), ctypes.c_void_p()
        whole, part, rest = (ctypes.create_string_buffer(144) for _ in range(3))  # CUdevResource
        # (dev, desc and green are read when their call is made: ctypes passes the objects' values then)
        for call, args in (("cuDeviceGet", (ctypes.byref(dev), 0)),
                           ("cuDeviceGetDevResource", (dev, whole, 1)),
                           ("cuDevSmResourceSplitByCount", (part, ctypes.byref(count), whole, rest, 0, sms)),
                           ("cuDevResourceGenerateDesc", (ctypes.byref(desc), part, 1)),
                           ("cuGreenCtxCreate", (ctypes.byref(self.green), desc, dev, 1)),
                           ("cuGreenCtxStreamCreate", (ctypes.byref(self.stream), self.green, 1, 0))):
            if not hasattr(self.lib, call) or getattr(self.lib, call)(*args) != 0:
                pytest.skip(f"{call}: no green contexts here")

    def close(self):
        self.lib.cuStreamDestroy_v2(self.stream)
        self.lib.cuGreenCtxDestroy(self.green)


# On a stream that may use a few of the SMs only, the run kernel's blocks have to
# fit those: they wait for one another.
def test_stream_on_part_of_the_gpu(cc):
    torch = pytest.importorskip("torch")
    ro, col, lab = _job(20011, 12)
    ref = oracle.sync_run(ro, col, lab, 20)
    torch.cuda.init()
    with cc.Consensus(ro, col, lab) as job:
        part = _Part(16)
        job.set_wait_limit(2 * SECOND)
        for stream in (part.stream.value, 0, part.stream.value):
            job.set_stream(stream)
            job.reset()
            assert job.run_until_converged(20) == ref.sweeps
            assert job.history() == ref.stats
            np.testing.assert_array_equal(job.cluster_ids(), ref.C)
        job.set_stream(0)
        dev = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (ro, col, lab)]
        torch.cuda.synchronize()
        with cc.Consensus.from_device(len(ro) - 1, len(col), dev[0].data_ptr(), dev[1].data_ptr(), len(lab),
                                      dev[2].data_ptr(), stream=part.stream.value) as other:
            other.set_wait_limit(2 * SECOND)
            assert other.run_until_converged(20) == ref.sweeps
            assert other.history() == ref.stats
        part.close()


# Up to 768 jobs one block takes the jobs' decisions, more are a step of all
# blocks; from random warm starts some jobs fall back to the matching.
@pytest.mark.parametrize("opts", [{}, {"active_set": 1}, {"colour_batched": 1}, {"sweep_mode": 1}, {"sweep_mode": 2}])
@pytest.mark.parametrize("count", [768, 769, 1100])
def test_many_jobs(cc, count, opts):
    rng = np.random.default_rng(count)
    kinds, starts = [], []
    for n, k in [(1, 1), (2, 3), (5, 2), (9, 5), (17, 4), (33, 7), (40, 3), (64, 6), (21, 9), (12, 12), (50, 5), (30, 2)] * 2:
        u = rng.integers(0, n, 3 * n)
        ro, col = csr_from_edges(n, u, (u + rng.integers(0, n, 3 * n)) % n)
        kinds.append((ro, col, rng.integers(0, 1 + n // 4, (k, n)).astype(np.int32)))
        starts.append(rng.integers(0, n, n).astype(np.int32) // 3 * 3)
    run = oracle.colour_run if opts.get("colour_batched") else oracle.sync_run
    warm = [run(*j, 20, C0=c) for j, c in zip(kinds, starts)]
    assert any(s["fallback"] for r in warm for s in r.stats)
    fresh = [run(*j, 20) for j in kinds]
    pick = rng.integers(0, len(kinds), count)
    with cc.ConsensusBatch([kinds[i] for i in pick], _options(cc, **opts)) as batch:
        for refs in (fresh, warm, fresh):
            batch.reset()
            if refs is warm:
                batch.set_cluster_ids(np.concatenate([starts[i] for i in pick]))
            batch.run_until_converged(20)
            np.testing.assert_array_equal(batch.cluster_ids(), np.concatenate([refs[i].C for i in pick]))
            for j, i in enumerate(pick):
                assert batch.history(j) == refs[i].stats


# Noisy labels: the first sweeps leave clusters of a few members that agree on
# little, so the table that follows a partial one holds most of their label rows.
@pytest.mark.parametrize("tight", [0, 1, 2])
@pytest.mark.parametrize("n,k,classes", [(100, 6, 4), (61, 9, 60), (300, 5, 2)])
def test_noisy_labels(cc, n, k, classes, tight):
    rng = np.random.default_rng(n)
    jobs = []
    for _ in range(40):
        u = rng.integers(0, n, 4 * n)
        ro, col = csr_from_edges(n, u, (u + rng.integers(1, max(2, n // 8), 4 * n)) % n)
        jobs.append((ro, col, rng.integers(0, classes, (k, n)).astype(np.int32)))
    refs = [oracle.sync_run(*j, 20) for j in jobs]
    with cc.ConsensusBatch(jobs, _options(cc, tight_rebuild=tight)) as batch:
        batch.run_until_converged(20)
        assert [batch.history(j) for j in range(len(jobs))] == [r.stats for r in refs]
        np.testing.assert_array_equal(batch.cluster_ids(), np.concatenate([r.C for r in refs]))


def _large_graph(rng, n):
    u = rng.integers(0, n, 50 * n)
    v = np.where(rng.random(len(u)) < 0.5, u // 120 * 120 + rng.integers(0, 120, len(u)), rng.integers(0, n, len(u)))
    return csr_from_edges(n, u, np.minimum(v, n - 1))


# Jobs that fill the GPU many times over (4 million CSR entries) run as graphs
# while others are in flight; the same runs in turn, at once, and mixed with
# small ones.
def test_large_runs_in_threads(cc):
    rng = np.random.default_rng(11)
    n = 60011
    large = _large_graph(rng, n)
    labs = [np.where(rng.random((5, n)) < 0.3, rng.integers(0, n // 120, (5, n)), np.arange(n) // 120).astype(np.int32)
            for _ in range(3)]
    jobs = [(*large, lab) for lab in labs] + [_job(6007, 9), _job(20011, 12)]
    refs = [oracle.sync_run(*j, 6) for j in jobs]
    wrong = []

    def work(i):
        with cc.Consensus(*jobs[i]) as job:
            for _ in range(8):
                job.reset()
                sweeps = job.run_until_converged(6)
                ms, prop = job.last_run_timing()
                if (sweeps, job.history()) != (refs[i].sweeps, refs[i].stats) or len(ms) != sweeps or \
                        not np.array_equal(job.cluster_ids(), refs[i].C):
                    wrong.append(i)

    for i in range(len(jobs)):
        work(i)
    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong


# A small job's run is a chain of small kernels; beside another thread's large runs
# it waits for their kernels, not for the end of a run with each of its own.
def test_small_run_beside_large_ones(cc):
    rng = np.random.default_rng(12)
    n = 60011
    lab = np.where(rng.random((12, n)) < 0.3, rng.integers(0, n // 120, (12, n)), np.arange(n) // 120).astype(np.int32)
    small_job = _job(1000, 10)
    ref = oracle.sync_run(*small_job, 20)
    stop = threading.Event()

    def runs(job):
        while not stop.is_set():
            job.reset()
            job.run_until_converged(6)

    def median(job, count):
        times = []
        for _ in range(count):
            t0 = time.perf_counter()
            job.reset()
            assert job.run_until_converged(20) == ref.sweeps
            times.append(time.perf_counter() - t0)
            np.testing.assert_array_equal(job.cluster_ids(), ref.C)
        return np.median(times)

    with cc.Consensus(*_large_graph(rng, n), lab) as large, cc.Consensus(*small_job) as small:
        large.run_until_converged(6)
        alone = median(small, 20)
        thread = threading.Thread(target=runs, args=(large,))
        thread.start()
        try:
            beside = median(small, 20)
        finally:
            stop.set()
            thread.join()
    assert beside < 15 * alone, (beside, alone)  # about 100 where each kernel waits for a run


# A small job's cc_sweep is a graph of one sweep: the kernels of one body outside
# its regions, and none of a second.
def test_single_sweeps_of_a_small_job(cc):
    ro, col, lab = _job(1000, 10)
    ref = oracle.sync_run(ro, col, lab, 20)
    outside = 17  # begin, own, edges, collect, route, 6 gates, bid, match keys, commit, match reset, end jobs, end
    with cc.Consensus(ro, col, lab) as job:
        for rounds in range(2):
            job.reset()
            for s in range(ref.sweeps):
                before = job.launch_count()
                assert job.sweep() == ref.stats[s]
                assert job.launch_count() - before >= 1 + outside
                assert len(job.last_run_timing()[0]) == 1
            assert job.launch_count() - before == 1 + outside  # the last one proposes nothing
            np.testing.assert_array_equal(job.cluster_ids(), ref.C)
            job.reset()
            assert job.run_until_converged(20) == ref.sweeps
            assert job.history() == ref.stats


# Batches and colour-batched jobs of that size beside another thread's runs: the
# graph of a run with several jobs, and with colour classes.
def test_large_batches_beside_runs(cc):
    rng = np.random.default_rng(13)
    n = 60011
    lab = np.where(rng.random((4, n)) < 0.3, rng.integers(0, n // 120, (4, n)), np.arange(n) // 120).astype(np.int32)
    large = (*_large_graph(rng, n), lab)
    jobs = [_job(900, 12), large, _job(3001, 5)]
    refs = [oracle.sync_run(*j, 5) for j in jobs]
    colour = oracle.colour_run(*large, 2)
    small_job = _job(1000, 10)
    stop = threading.Event()

    def runs():
        with cc.Consensus(*small_job) as small:
            while not stop.is_set():
                small.reset()
                small.run_until_converged(20)

    thread = threading.Thread(target=runs)
    thread.start()
    graphs = 0
    try:
        with cc.ConsensusBatch(jobs) as batch, cc.Consensus(*large, _options(cc, colour_batched=1)) as coloured, \
                cc.ConsensusBatch(jobs, _options(cc, active_set=1, debug_checks=1)) as active:
            for _ in range(4):
                for b in (batch, active):
                    before = b.launch_count()
                    b.reset()
                    b.run_until_converged(5)
                    graphs += b.launch_count() - before > 20
                    np.testing.assert_array_equal(b.cluster_ids(), np.concatenate([r.C for r in refs]))
                    assert [b.history(j)[-1] for j in range(3)] == [r.stats[-1] for r in refs]
                before = coloured.launch_count()
                coloured.reset()
                coloured.run_until_converged(2)
                graphs += coloured.launch_count() - before > 20
                assert coloured.history() == colour.stats
                np.testing.assert_array_equal(coloured.cluster_ids(), colour.C)
    finally:
        stop.set()
        thread.join()
    assert graphs > 0

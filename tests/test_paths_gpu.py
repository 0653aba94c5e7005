"""The GPU paths that are chosen by size, at the sizes where the choice
changes, against the oracle (whole numbers exact; variation of information
within the rounding of its fp64 sums of at most n log n)."""
import numpy as np
import pytest

import oracle
from workloads import make_config
from workloads.graphs import csr_from_edges

pytestmark = pytest.mark.gpu

VI_TOL = 1e-9  # nats; see test_metrics_gpu.py


@pytest.fixture(scope="module")
def cc():
    import __graft_entry__

    __graft_entry__.build()
    import paper_2408_11331_gb300 as m

    return m


def _graph(rng, n):
    u = rng.integers(0, n, 4 * n)
    return csr_from_edges(n, u, (u + rng.integers(1, max(2, n // 8), 4 * n)) % n)


# matrices of 16 n + 2^18 cells at most are counted densely: with n = 1000, up
# to 527 classes; a partition of singletons or of 528 classes takes the tables
@pytest.mark.parametrize("n,classes", [(1, [1]), (2, [1, 2]), (33, [1, 33, 7]), (1000, [527, 1, 500, 3, 32]),
                                       (1000, [528, 2, 9]), (1021, [1021, 4, 4, 4, 4, 4, 4, 60, 1]),
                                       (5003, [40] * 13)])
def test_partition_distances(cc, n, classes):
    rng = np.random.default_rng(n + len(classes))
    lab = np.stack([np.where(np.arange(n) < K, np.arange(n), rng.integers(0, K, n)) for K in classes]).astype(np.int32)
    lab[0] = -lab[0]  # any int32 values
    ro, col = _graph(rng, n) if n > 1 else (np.zeros(2, np.int64), np.empty(0, np.int32))
    with cc.Consensus(ro, col, lab) as job:
        before = job.cluster_ids()
        got = job.partition_distances()
        np.testing.assert_array_equal(job.cluster_ids(), before)
        metrics = job.metrics()
        want0 = oracle.metrics(lab, oracle.singletons(n))
        for f in ("mirkin", "split_join"):
            np.testing.assert_array_equal(metrics[f], want0[f])
    for a in range(len(classes)):
        first = {}
        C = np.array([first.setdefault(x, v) for v, x in enumerate(lab[a])], np.int32)
        want = oracle.metrics(lab, C)
        for f in ("mirkin", "split_join"):
            np.testing.assert_array_equal(got[f][a], want[f])
        np.testing.assert_allclose(got["rand_distance"][a], want["rand_distance"], rtol=1e-14, atol=0)
        np.testing.assert_allclose(got["vi"][a], want["vi"], rtol=0, atol=VI_TOL)


# 16,384 label rows is where a single job moves to the run kernel; the k cover
# whole and ragged quads of partitions, one lane and several per item
@pytest.mark.parametrize("n,k", [(5461, 3), (5462, 3), (4096, 4), (1365, 12), (1366, 11), (700, 33), (3001, 65)])
@pytest.mark.parametrize("opts", [{}, {"active_set": 1}, {"empty_moves": 1}, {"lanes": 1}, {"lanes": 32},
                                  {"tight_rebuild": 2}, {"no_regions": 1}])
def test_sweeps_around_the_run_kernel(cc, n, k, opts):
    c = make_config("lfr", n=n, k=k, cmin=10, cmax=300, max_deg=100, seed=n + k)
    ro, col, lab = c["row_off"], c["col"], c["labels"]
    ref = oracle.sync_run(ro, col, lab, 20, empty=bool(opts.get("empty_moves")))
    o = cc.cc_default_options()
    for f, x in opts.items():
        setattr(o, f, x)
    with cc.Consensus(ro, col, lab, o) as job:
        for _ in range(2):
            job.reset()
            assert job.run_until_converged(20) == ref.sweeps
            assert job.history() == ref.stats
            np.testing.assert_array_equal(job.cluster_ids(), ref.C)
            assert job.objective_recompute() == ref.F
            ms, prop = job.last_run_timing()
            assert len(ms) == ref.sweeps and np.all(prop > 0) and np.all(prop <= ms)
        job.reset()  # sweep by sweep: host calls between a partial table and the next sweep
        for s in range(3):
            job.sweep()
            job.metrics()
            assert job.objective_recompute() == ref.stats[min(s, ref.sweeps - 1)]["F"]
        job.run_until_converged(20)
        np.testing.assert_array_equal(job.cluster_ids(), ref.C)


# many classes (more than the first label map takes: 2^16 entries, or a quarter
# of the labels), one class, and a mix, against the oracle's run
@pytest.mark.parametrize("n,k,kinds", [(30011, 6, "sssooo"), (70003, 2, "ss"), (1023, 3, "oso"), (1025, 5, "soooo")])
def test_label_maps(cc, n, k, kinds):
    rng = np.random.default_rng(n)
    lab = np.stack([rng.permutation(n).astype(np.int32) - n // 2 if q == "s" else (np.arange(n) // 37).astype(np.int32)
                    for q in kinds])
    ro, col = _graph(rng, n)
    ref = oracle.sync_run(ro, col, lab, 4)
    with cc.Consensus(ro, col, lab) as job, cc.ConsensusBatch([(ro, col, lab), (ro, col, lab[:1])]) as batch:
        job.run_until_converged(4)
        assert job.history() == ref.stats
        np.testing.assert_array_equal(job.cluster_ids(), ref.C)
        batch.run_until_converged(4)
        assert batch.history(0) == ref.stats
        np.testing.assert_array_equal(batch.cluster_ids()[:n], ref.C)


# one, two and all vertices per neighbour list: windows of the scoring with 128
# distinct vertices, with 64, and with one
@pytest.mark.parametrize("shape", ["matching", "ring", "star"])
@pytest.mark.parametrize("n,k", [(1000, 3), (5000, 9)])
def test_sparse_graphs(cc, shape, n, k):
    rng = np.random.default_rng(n + k)
    v = np.arange(n)
    if shape == "matching":
        ro, col = csr_from_edges(n, v[::2], v[1::2])
    elif shape == "ring":
        ro, col = csr_from_edges(n, v, (v + 1) % n)
    else:
        ro, col = csr_from_edges(n, np.zeros(n - 1, np.int64), v[1:])
    lab = np.stack([(v // rng.integers(2, 40) + (rng.random(n) < 0.1) * 7).astype(np.int32) for _ in range(k)])
    ref = oracle.sync_run(ro, col, lab, 20)
    for opts in ({}, {"active_set": 1}, {"no_regions": 1}):
        o = cc.cc_default_options()
        for f, x in opts.items():
            setattr(o, f, x)
        with cc.Consensus(ro, col, lab, o) as job:
            job.run_until_converged(20)
            assert job.history() == ref.stats
            np.testing.assert_array_equal(job.cluster_ids(), ref.C)


# 16-bit label rows hold partitions of up to 65535 classes, and up to 512
# partitions are counted in shared memory: both sides of both lines, alone and
# next to a job of the other kind
@pytest.mark.parametrize("n,classes", [(66001, [65535, 900, 65534]), (66001, [900, 65536, 900]), (301, [40] * 512),
                                       (301, [40] * 513)])
def test_label_rows(cc, n, classes):
    rng = np.random.default_rng(len(classes) + classes[0])
    base = np.arange(n) // 33
    lab = np.stack([np.where(np.arange(n) < K, np.arange(n), rng.integers(0, K, n)) if K > 1000 else
                    np.where(rng.random(n) < 0.2, rng.integers(0, K, n), base % K) for K in classes]).astype(np.int32)
    ro, col = _graph(rng, n)
    small = make_config("lfr", n=2000, k=9, cmin=10, cmax=300, max_deg=100, seed=n)
    jobs = [(ro, col, lab), (small["row_off"], small["col"], small["labels"])]
    refs = [oracle.sync_run(*j, 6) for j in jobs]
    with cc.Consensus(*jobs[0]) as job, cc.ConsensusBatch(jobs) as batch:
        job.run_until_converged(6)
        assert job.history() == refs[0].stats
        np.testing.assert_array_equal(job.cluster_ids(), refs[0].C)
        want, got = oracle.metrics(lab, refs[0].C), job.metrics()
        for f in ("mirkin", "split_join"):
            np.testing.assert_array_equal(got[f], want[f])
        batch.run_until_converged(6)
        assert [batch.history(j) for j in range(2)] == [r.stats for r in refs]
        np.testing.assert_array_equal(batch.cluster_ids(), np.concatenate([r.C for r in refs]))

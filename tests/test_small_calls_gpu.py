"""Calls whose way depends on how small the job is, on both sides of each line,
against the oracle (whole numbers exact; variation of information within the
rounding of its fp64 sums of at most n log n)."""
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


def _same(got, want):
    for f in ("mirkin", "split_join"):
        np.testing.assert_array_equal(got[f], want[f])
    np.testing.assert_allclose(got["rand_distance"], want["rand_distance"], rtol=1e-14, atol=0)
    np.testing.assert_allclose(got["vi"], want["vi"], rtol=0, atol=VI_TOL)


# Tables of 2^16 slots and of 2^17 (counts tallied first), and scratch below and
# above the megabyte that a context keeps; every call twice, the second on what
# the first left.
@pytest.mark.parametrize("n,k,distinct", [(10, 3, False), (2000, 10, False), (4000, 10, False), (4000, 10, True),
                                          (30011, 9, True)])
def test_metrics_small_and_large(cc, n, k, distinct):
    rng = np.random.default_rng(n + k)
    base = np.arange(n) // 90
    lab = np.stack([rng.permutation(n) if distinct else np.where(rng.random(n) < 0.2, rng.integers(0, 9, n), base)
                    for _ in range(k)]).astype(np.int32)
    with cc.Consensus(*_graph(rng, n), lab) as job:
        for C in (None, base * 90, rng.integers(0, n, n)):
            if C is not None:
                job.set_cluster_ids(C.astype(np.int32))
            want = oracle.metrics(lab, oracle.singletons(n) if C is None else C.astype(np.int32))
            for _ in range(2):
                _same(job.metrics(), want)


# The objective between sweeps, where the table holds the clusters of more than 8
# members only, without rebuilding it; ragged k, several lanes and one.
@pytest.mark.parametrize("n,k", [(20011, 12), (6007, 9), (1000, 10), (3001, 33), (40, 3)])
def test_objective_after_a_partial_table(cc, n, k):
    c = make_config("lfr", n=n, k=k, cmin=10, cmax=300, max_deg=100, seed=n + k)
    ro, col, lab = c["row_off"], c["col"], c["labels"]
    ref = oracle.sync_run(ro, col, lab, 20)
    with cc.Consensus(ro, col, lab) as job:
        for s in range(ref.sweeps):
            job.sweep()
            before = job.table_stats()
            assert job.objective_recompute() == ref.stats[s]["F"]
            assert job.table_stats() == before
        np.testing.assert_array_equal(job.cluster_ids(), ref.C)
    o = cc.cc_default_options()
    o.debug_checks = 1  # the same sums, job by job
    with cc.ConsensusBatch([(ro, col, lab), (ro, col, lab[:1]), (ro, col, lab[::2])], o) as batch:
        for s in range(3):
            batch.sweep()


# Sizes and member lists of a warm start are counted in tiles of 256 vertices, of
# 1024 above 2^17 vertices: tile edges, one cluster, many, and two large ones.
@pytest.mark.parametrize("n", [1, 255, 256, 257, 1025, (1 << 17) - 1, 1 << 17, (1 << 17) + 1])
def test_warm_start_tiles(cc, n):
    rng = np.random.default_rng(n)
    lab = np.stack([np.arange(n) // 50, rng.integers(0, 40, n), np.arange(n) % 7]).astype(np.int32)
    ro, col = _graph(rng, n) if n > 1 else (np.zeros(2, np.int64), np.empty(0, np.int32))
    with cc.Consensus(ro, col, lab) as job:
        for C in (np.zeros(n), np.arange(n)[::-1], rng.integers(0, n, n), np.where(rng.random(n) < 0.9, n - 1, 0)):
            C = C.astype(np.int32)
            job.set_cluster_ids(C)
            assert job.objective() == oracle.objective(lab, C) == job.objective_recompute()
            np.testing.assert_array_equal(job.cluster_ids(), C)
            assert job.run_until_converged(1) == 1
            step = oracle.sync_step(ro, col, lab, C)
            np.testing.assert_array_equal(job.cluster_ids(), step.C)
            assert job.history()[-1] == step.stats


# Dense graphs are assembled in slices of their vertices' entries: cliques and a
# graph whose rows are partly empty, alone and behind another job.
@pytest.mark.parametrize("n,full", [(33, 33), (65, 64), (700, 700), (1500, 1500), (2100, 900)])
def test_dense_graphs(cc, n, full):
    rng = np.random.default_rng(n)
    u, v = np.triu_indices(full, 1)
    ro, col = csr_from_edges(n, u, v)
    lab = (np.arange(n)[None, :] // np.array([[7], [9], [40]]) + (rng.random((3, n)) < 0.2)).astype(np.int32)
    ref = oracle.sync_run(ro, col, lab, 6)
    other = (*_graph(rng, 50), rng.integers(0, 9, (2, 50)).astype(np.int32))
    with cc.Consensus(ro, col, lab) as job, cc.ConsensusBatch([other, (ro, col, lab)]) as batch:
        job.run_until_converged(6)
        assert job.history() == ref.stats
        np.testing.assert_array_equal(job.cluster_ids(), ref.C)
        batch.run_until_converged(6)
        assert batch.history(1) == ref.stats
        np.testing.assert_array_equal(batch.cluster_ids()[50:], ref.C)
    bad = col.copy()
    bad[len(bad) // 2] = n
    with pytest.raises(cc.CCError) as e:
        cc.Consensus(ro, bad, lab)
    assert e.value.status == 1


# More classes than the first label map holds (2^16 entries, or a quarter of the
# labels): the compaction stops and runs again, and the sums over the classes are
# those of the second run.
@pytest.mark.parametrize("n,k,distinct", [(70001, 3, 3), (70001, 3, 1), (30011, 9, 9), (30011, 9, 2)])
def test_label_map_runs_again(cc, n, k, distinct):
    rng = np.random.default_rng(n + distinct)
    lab = np.stack([rng.permutation(n) if i < distinct else np.arange(n) // 41 for i in range(k)]).astype(np.int32)
    other = (*_graph(rng, 500), rng.integers(0, 30, (4, 500)).astype(np.int32))
    mine = (*_graph(rng, n), lab)
    C = (np.arange(n) // 60 * 60).astype(np.int32)
    with cc.Consensus(*mine) as job, cc.ConsensusBatch([other, mine]) as batch:
        job.set_cluster_ids(C)
        _same(job.metrics(), oracle.metrics(lab, C))
        assert job.objective() == oracle.objective(lab, C)
        batch.set_cluster_ids(np.concatenate([np.zeros(500, np.int32), C]))
        got = batch.metrics()
        _same(got[0], oracle.metrics(other[2], np.zeros(500, np.int32)))
        _same(got[1], oracle.metrics(lab, C))
        assert batch.objective(1) == oracle.objective(lab, C)

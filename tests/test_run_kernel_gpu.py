"""The run kernel beside the ordinary run: waits that run out, against the
oracle (whole numbers, exact)."""
import numpy as np
import pytest

import oracle
from workloads import make_config

pytestmark = pytest.mark.gpu

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

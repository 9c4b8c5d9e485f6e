"""The per-walk tour sums X_n are zero between launches: a tour that has ended leaves none
behind, whatever walks its parts grew on.

Each test grows a run that may leave something, resets it, and grows simple chains
(cut-offs that are never active: no copies, so the run depends on its streams alone) on
the same rows: their W_n and Q_n equal the oracle's.  Sums left in a row would be added to
the next tour of that row and show in Q_n (one of 1200 tours: 1e-3 and more, against the
1e-12 allowed for the order of the sums)."""
import numpy as np
import pytest

from oracle import oracle as orc
from tests.gpu_util import REL_W, Run, torch_cuda

pytestmark = pytest.mark.gpu


def _chains(d, n_max, N, seed, tours):
    o = orc.Oracle(d, n_max, N, seed=seed)
    o.set_cutoffs(np.full(n_max + 1, np.inf), np.zeros(n_max + 1), 2, 2.0)
    o.run(tours)
    return o.tables()


def _grow_chains(run, n_max, tours):
    run.set_cutoffs(np.full(n_max + 1, np.inf), np.zeros(n_max + 1), 2, 2.0)
    run.run(tours)
    return run.tables()


def _same(g, t):
    close = lambda a, b: np.all(np.abs(a - b) <= REL_W * np.maximum(np.abs(a), np.abs(b)))
    assert np.array_equal(g["S"], t["S"])
    assert close(g["W"], t["W"])
    assert close(g["Q"], t["Q"])


@pytest.mark.parametrize("d,n_max,N", [(2, 24, 400), (3, 60, 400), (3, 60, 1500)])
def test_shared_tours_leave_no_sums_behind(d, n_max, N):
    torch_cuda()
    t = _chains(d, n_max, N, 29, 3)
    with Run(d, n_max, N, 29) as run:
        for _ in range(4):
            run.set_cutoffs(None, None)
            run.run(30)
            st = run.stats()
            assert st["status"] == 0 and st["shared"] > 0
            assert st["tours_finished"] == 30 * N
            run.reset()
            _same(_grow_chains(run, n_max, 3), t)
            run.reset()


def test_a_reset_clears_a_failed_run_that_nobody_asked_about():
    """A queued run that stops at its time bound, a reset with no query between, and the
    next run starts from zero tour sums all the same."""
    torch_cuda()
    d, n_max, N = 3, 60, 400
    t = _chains(d, n_max, N, 31, 3)
    # 400 x 4000 tours of some 60 nodes, 9.6e7 nodes: tens of ms, against a bound of 5 ms
    with Run(d, n_max, N, 31, max_seconds=0.005) as run:
        for _ in range(2):
            run.set_cutoffs(None, None)
            run.run(4000, sync=False)
            run.reset()
            _same(_grow_chains(run, n_max, 3), t)
            assert run.stats()["status"] == 0
            run.reset()

"""The admission of tours under cut-offs: none by default (cut-offs read no table), and the
caller's limit where one was given, also one that equals flatPERM's default, and also
after a checkpoint.

304 chains of one tour each: without a limit all grow at once; with at most
2 + 0.25 x finished in flight they take some 20 generations, one after another.  Asserted
is a factor of 4 in time either way."""
import time

import numpy as np
import pytest

import paper_2002_03000_gb300 as pg
from tests.gpu_util import Run, torch_cuda

pytestmark = pytest.mark.gpu

D, N_MAX, N = 3, 500, 304


def _chains(run):
    run.set_cutoffs(np.full(N_MAX + 1, np.inf), np.zeros(N_MAX + 1), 2, 2.0)


def _seconds(run):
    best = np.inf
    for _ in range(4):
        run.reset()
        run.stats()
        t0 = time.perf_counter()
        run.run(1)
        best = min(best, time.perf_counter() - t0)
    return best


@pytest.mark.parametrize("given", [dict(ramp_c0=2, ramp_gamma=0.25), dict(ramp_c0=2), dict(ramp_gamma=0.25)])
def test_a_given_limit_holds_under_cutoffs(tmp_path, given):
    torch_cuda()
    path = str(tmp_path / "run.ckpt")
    with Run(D, N_MAX, N, 7, share_copies=-1) as run:
        _chains(run)
        free = _seconds(run)
        run.save(path)
    with pg.Run.load(path) as run:
        assert _seconds(run) < 2.0 * free
    with Run(D, N_MAX, N, 7, share_copies=-1, **given) as run:
        _chains(run)
        assert _seconds(run) > 4.0 * free
        run.save(path)
    with pg.Run.load(path) as run:
        assert _seconds(run) > 4.0 * free

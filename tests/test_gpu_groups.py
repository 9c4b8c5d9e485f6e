"""Walks held by groups of lanes, at the edges of the launch forms.

Runs whose tables do not depend on the schedule (cut-offs without sharing,
Algorithm 1, a single fresh sequence) equal the oracle's at any layout: the
shortest walks, more or fewer walks than a warp holds, walks in the arena, the
last cubic length with 32-bit keys and the first with 64-bit ones.  Counts exactly, weight
sums to relative 1e-12: only the order of the sums differs, and no length gets
more than 4000 positive terms here (k of them agree to k 2^-53, 4.5e-13)."""
import math

import numpy as np
import pytest

import paper_2002_03000_gb300 as pg
from oracle import oracle as orc
from paper_2002_03000_gb300 import batch as pb
from tests import inputs
from tests.gpu_util import REL_W, Run, torch_cuda

pytestmark = pytest.mark.gpu

FRESH, SNAP = pg.PERM_THRESH_FRESH, pg.PERM_THRESH_SNAPSHOT


def _cuts(d, n_max, f):
    return inputs.perm_cutoffs(d, n_max, f, lambda k: orc.scale_exp(d, k))


def _same(g, t, st):
    close = lambda a, b: np.all(np.abs(a - b) <= REL_W * np.maximum(np.abs(a), np.abs(b)))
    assert st["status"] == 0
    assert np.array_equal(g["M"], t["M"])
    assert np.array_equal(g["S"], t["S"])
    assert close(g["W"], t["W"]) and close(g["Q"], t["Q"])
    assert st["steps"] == t["steps"]


# (d, n_max, sequences, tours, layout)
LAYOUTS = [
    (2, 1, 5, 3, dict(threshold=SNAP)),
    (3, 1, 5, 3, dict(threshold=FRESH)),
    (2, 2, 33, 4, dict(threshold=FRESH, lanes_per_warp=32)),
    (3, 3, 33, 4, dict(threshold=SNAP, lanes_per_warp=1)),
    (2, 63, 77, 6, dict(threshold=SNAP, lanes_per_warp=3, slots=50)),
    (3, 63, 77, 6, dict(threshold=FRESH, lanes_per_warp=3, max_ctas=2)),
    (2, 400, 1100, 2, dict(threshold=SNAP)),                    # flatPERM: four copies of the tables
    (2, 401, 1100, 2, dict(threshold=SNAP)),                    # one
    (2, 400, 1100, 2, dict(threshold=SNAP, slots=511)),
    (3, 100, 700, 3, dict(threshold=SNAP, observables=1)),      # watched
    (3, 512, 40, 3, dict(threshold=SNAP, stack_ring=128)),      # 32-bit keys
    (3, 513, 40, 3, dict(threshold=SNAP, hash_scale=1)),        # 64-bit keys
    (2, 90, 40, 5, dict(threshold=SNAP, walk_memory=2)),        # walks in the arena
    (3, 600, 20, 3, dict(threshold=FRESH, walk_memory=2, hash_scale=2)),
    (2, 40, 90, 4, dict(threshold=SNAP, max_ctas=1)),           # one full CTA: 88 walks, 44, 13
    (3, 40, 50, 4, dict(threshold=FRESH, max_ctas=1)),
    (3, 513, 30, 2, dict(threshold=SNAP, max_ctas=1, lanes_per_warp=2)),
    (2, 63, 77, 6, dict(threshold=SNAP, ramp_c0=3)),            # an admission limit of the caller's
    (2, 300, 60, 2, dict(threshold=SNAP, max_ctas=-1)),
]


@pytest.mark.parametrize("d,n_max,N,tours,layout", LAYOUTS)
def test_cutoff_runs_equal_the_oracle_at_any_layout(d, n_max, N, tours, layout):
    torch_cuda()
    hi, lo = _cuts(d, n_max, 1.4)
    o = orc.Oracle(d, n_max, N, seed=23)
    o.set_cutoffs(hi, lo, 2, 2.0)
    o.run(tours)
    with Run(d, n_max, N, 23, share_copies=-1, **layout) as run:
        run.set_cutoffs(hi, lo, 2, 2.0)
        run.run(tours - 1)                       # the sums continue over launches
        run.run(1)
        _same(run.tables(), o.tables(), run.stats())


def test_odd_cutoffs_equal_the_oracle():
    """Cut-offs that no weight is compared with as usual: NaN, zeros of both signs,
    negative numbers, infinities, subnormals."""
    torch_cuda()
    d, n_max, N = 2, 40, 30
    hi, lo = _cuts(d, n_max, 1.4)
    hi[20:29] = [math.nan, 30.0, -math.nan, 30.0, 0.0, 30.0, -0.0, math.inf, -1.0]
    lo[5:19] = [math.nan, 0.1, -math.nan, 0.1, 0.0, 0.1, -0.0, 0.1, -1.0, 0.1, -math.inf, 0.1, 5e-324, 0.1]
    o = orc.Oracle(d, n_max, N, seed=5)
    o.set_cutoffs(hi, lo, 2, 2.0)
    o.run(4)
    with Run(d, n_max, N, 5, threshold=FRESH) as run:
        run.set_cutoffs(hi, lo, 2, 2.0)
        run.run(4)
        _same(run.tables(), o.tables(), run.stats())


# a sequence's own rows through L1 (Algorithm 1, one sequence), plain and watched
FRESH_RUNS = [
    (2, 1, 3, 5, dict(alg=pg.PERM_ALG1)),
    (2, 17, 41, 30, dict(alg=pg.PERM_ALG1, lanes_per_warp=8)),
    (3, 12, 41, 20, dict(alg=pg.PERM_ALG1, lanes_per_warp=4, max_ctas=3, observables=1)),
    (2, 5, 1, 200, dict(threshold=FRESH)),
    (3, 40, 1, 100, dict(threshold=FRESH, walk_memory=2)),
    (2, 33, 1, 100, dict(threshold=FRESH, observables=1)),
]


@pytest.mark.parametrize("d,n_max,N,tours,layout", FRESH_RUNS)
def test_fresh_runs_equal_the_oracle(d, n_max, N, tours, layout):
    torch_cuda()
    o = orc.Oracle(d, n_max, N, seed=31, alg=orc.ORC_ALG1 if "alg" in layout else orc.ORC_ALG2)
    o.run(tours)
    with Run(d, n_max, N, 31, **layout) as run:
        run.run(tours - 2)
        run.run(2)
        _same(run.tables(), o.tables(), run.stats())


@pytest.mark.parametrize("d,n_max,N,tours,layout", [
    (2, 3, 2, 50, dict()),                                       # fewer walks than a warp holds
    (2, 20, 9, 400, dict(threshold=FRESH)),                      # a row that several walks add to
    (2, 400, 600, 3, dict()),
    (2, 30, 600, 20, dict(observables=1)),                       # watched
    (3, 513, 64, 4, dict(walk_memory=2)),
    (3, 20, 100, 10, dict(helper_walks=64)),
])
def test_interacting_runs_keep_what_holds_for_any_schedule(d, n_max, N, tours, layout):
    """Every tour is counted at lengths 0 and 1 and every node once, and c_1 = 2d."""
    torch_cuda()
    with Run(d, n_max, N, 3, **layout) as run:
        run.run(tours)
        lc, S, rv = run.estimates()
        st = run.stats()
    assert st["status"] == 0 and st["tours_finished"] == N * tours
    assert S[0] == N * tours and S[1] == N * tours
    assert int(S.sum()) == st["steps"]
    assert math.isclose(math.exp(lc[1]), 2 * d, rel_tol=1e-12)


def test_flatperm_after_cutoffs_without_an_admission_limit():
    """Cut-offs admit every tour at once; the limit holds again for flatPERM after them."""
    torch_cuda()
    d, n_max, N = 2, 100, 700
    hi, lo = _cuts(d, n_max, 1.4)
    with Run(d, n_max, N, 12) as run:
        for k in (1, 2):
            run.set_cutoffs(hi, lo, 2, 2.0)
            run.run(2)
            run.set_cutoffs(None, None)
            run.run(3)
            lc, S, rv = run.estimates()
            st = run.stats()
            assert st["status"] == 0 and st["tours_finished"] == 5 * k * N
            assert S[0] == S[1] == 5 * k * N and int(S.sum()) == st["steps"]
            assert math.isclose(math.exp(lc[1]), 2 * d, rel_tol=1e-12)


@pytest.mark.parametrize("runs", [1, 512, 513])
def test_persistent_batches_of_tiny_runs_complete(runs):
    """One run; the most runs whose CTAs are shared out at the start; one more."""
    torch_cuda()
    cfgs = [pb.make_config(2 + i % 2, 4 + i % 3, 1 + i % 5, 9, run_id=i, max_seconds=60.0) for i in range(runs)]
    with pb.Batch(cfgs, [2] * runs, persistent=True) as b:
        b.run()
        for r, cfg in enumerate(cfgs):
            lc, S, rv = b.estimates(r)
            st = b.stats(r)
            assert st["status"] == 0 and st["tours_finished"] == 2 * cfg.n_seq
            assert S[0] == S[1] == 2 * cfg.n_seq and int(S.sum()) == st["steps"]
            assert math.isclose(math.exp(lc[1]), 2 * cfg.d, rel_tol=1e-12)

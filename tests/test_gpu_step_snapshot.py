"""Step parity of the snapshot form (the states and the comparison of test_gpu_step, which
covers the fresh form): decisions and steps exactly, r bit for bit where the kernel
evaluated it exactly, child weights to relative 1e-12, on random states and on states
next to every decision boundary, on the kernel's own path and with every r exact."""
import numpy as np
import pytest

from tests import gpu_util, inputs, test_gpu_step as fresh
from paper_2002_03000_gb300 import _native as nat

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def snapshot_form(monkeypatch):
    """debug_step of the helpers goes through the snapshot form's entry point."""
    monkeypatch.setattr(gpu_util.nat, "perm_debug_step", nat.perm_debug_step_snapshot)


@pytest.mark.parametrize("d,n_max", [(2, 1), (2, 512), (3, 30), (3, 512)])
@pytest.mark.parametrize("force_exact", [0, 1])
def test_random_states(d, n_max, force_exact):
    states = inputs.snapshot_batch(300 + d * 7 + n_max, d, min(n_max, 200), 1500)
    fresh._compare(states, d, n_max, seed=0x1234ABCD5678EF01, force_exact=force_exact)


@pytest.mark.parametrize("d", [2, 3])
@pytest.mark.parametrize("force_exact", [0, 1])
def test_decision_boundaries(d, force_exact):
    seed = 0x0DDBA11
    states = fresh._boundary_states(np.random.default_rng(20 + d), d, 64, seed, 2000)
    exact = fresh._compare(states, d, 64, seed, force_exact=force_exact)
    assert np.mean(exact) > 0.9, np.mean(exact)


@pytest.mark.parametrize("d", [2, 3])
def test_edge_cases(d):
    fresh.test_step_parity_edge_cases(d)


@pytest.mark.parametrize("d,n_max", [(2, 30), (3, 24)])
def test_a_survivor_on_its_own_tour_number_is_divided_out(d, n_max):
    """Until a snapshot counts a tour, its nodes take the tour's own number for M, and a
    survivor's weight is the quotient (Wsum + W)/M, correctly rounded, times a_+ 2^-dE.
    Only the tour started last before a refresh has a number that is also a snapshot's
    (its survivors may take the product with 1/M): one of those that 64 walks start from
    one refresh, a quarter of a millisecond or more, to the next, 64 or more."""
    from oracle import oracle as orc
    gpu_util.torch_cuda()
    N = 64
    with gpu_util.Run(d, n_max, N, 77, refresh_ns=1000000, share_copies=-1) as run:
        run.trace_enable(1, 1, 40000)
        run.run(200)
        assert run.stats()["status"] == 0
        _, recs, _ = run.trace_read()
    own = [r for r in recs if r.c == 1 and r.n > 0 and r.r < 1.0 and not r.exact and r.M == r.tour * N + r.seq + 1]
    assert len(own) > 500
    same = 0
    for r in own:
        dE = orc.scale_exp(d, r.n + 1) - orc.scale_exp(d, r.n)
        same += r.child_w == (r.Wsum + r.W) / float(r.M) * (r.a_plus * 2.0 ** -dE)
    assert same >= 0.98 * len(own), (same, len(own))

"""The four copies of W_n and Q_n that the CTAs of a run with few lengths and many walks
add to (n_max <= 400, at least 512 walks), summed by the refresher and folded after a launch.

To n_max = 2 every tour has the same sums whatever the schedule: a node of length 1 carries
W = 2d, the table holds no more tours than M counts, so r >= 1 and nothing is pruned, and the
children of an enrichment share the node's weight.  So W_n = M c_n and Q_n = M c_n^2 at the
stored scale: bit for bit on the square lattice (integers over powers of two), to 1e-12 on
the cubic one (4800 terms, 4800 2^-53 = 5.3e-13).  A copy lost or counted twice shows in
either."""
import numpy as np
import pytest

from oracle import oracle as orc
from tests.gpu_util import REL_W, Run, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,layout", [(2, {}), (3, {}), (2, dict(share_copies=-1)), (3, dict(observables=1)),
                                      (2, dict(slots=511))])     # (511 walks: one copy)
def test_tables_of_equal_tours(d, layout):
    torch_cuda()
    N, n_max = 600, 2
    c = np.array([1.0, 2 * d, 2 * d * (2 * d - 1)]) * [2.0 ** -orc.scale_exp(d, k) for k in range(n_max + 1)]
    with Run(d, n_max, N, 19, **layout) as run:
        M = 0
        for tours in (1, 5, 2):                          # the sums continue over launches
            run.run(tours)
            M += tours * N
            t = run.tables()
            assert run.stats()["status"] == 0 and t["M"][0] == M
            if d == 2:
                assert np.array_equal(t["W"], M * c) and np.array_equal(t["Q"], M * c * c)
            assert np.all(np.abs(t["W"] - M * c) <= REL_W * M * c)
            assert np.all(np.abs(t["Q"] - M * c * c) <= REL_W * M * c * c)
        run.reset()
        run.run(1)
        t = run.tables()
        assert np.all(np.abs(t["W"] - N * c) <= REL_W * N * c) and np.all(np.abs(t["Q"] - N * c * c) <= REL_W * N * c * c)

"""Dense packing (max_ctas = -1): as few CTAs as hold one walk per sequence.  Numbers of
sequences just past what a CTA's layout holds, which can be fewer walks than its shared
memory has room for (n_max 400: 45 fit, 11 warps of 4 are taken)."""
import pytest

from tests.gpu_util import Run, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,n_max,layout", [(2, 400, {}), (2, 400, dict(lanes_per_warp=3)), (2, 64, {}),
                                            (3, 512, {}), (3, 1000, {}), (2, 90, dict(walk_memory=2))])
def test_every_sequence_has_its_walk(d, n_max, layout):
    torch_cuda()
    with Run(d, n_max, 100000, 1, max_ctas=1, **layout) as run:
        full = run.stats()["slots"]              # walks of one CTA
    for N, ctas in ((full - 1, 1), (full, 1), (full + 1, 2), (3 * full, 3), (3 * full + 1, 4)):
        with Run(d, n_max, N, 1, max_ctas=-1, **layout) as run:
            run.run(1)
            st = run.stats()
        assert st["status"] == 0 and st["tours_finished"] == N
        assert (st["slots"], st["ctas"]) == (N, ctas), (N, st)

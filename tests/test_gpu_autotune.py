"""The autotuner compares layouts, each once: a pick other than the default is a layout
of its own, never the default's under another name (lanes_per_warp past what a warp
holds, hash_scale 1 where 0 doubles the hash by itself)."""
import pytest

import paper_2002_03000_gb300 as pg
from paper_2002_03000_gb300 import batch as pb
from tests.gpu_util import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,n_max,N", [(2, 40, 900), (3, 40, 900), (2, 64, 64), (3, 20, 3000), (3, 600, 300), (2, 300, 64)])
def test_a_pick_is_a_layout_of_its_own(d, n_max, N):
    torch_cuda()

    def layout(**kw):
        with pg.Run(d, n_max, N, 3, **kw) as run:
            st = run.stats()
        return st["warps_per_cta"], st["lanes_per_warp"], st["hash_slots"], kw.get("stack_ring", 16)

    cfg = pb.make_config(d, n_max, N, 3, max_seconds=60.0)
    pb.autotune(cfg, probe_tours=1)
    pick = dict(lanes_per_warp=cfg.lanes_per_warp, hash_scale=cfg.hash_scale, stack_ring=cfg.stack_ring)
    assert cfg.stack_ring in (16, 64)
    if (cfg.lanes_per_warp, cfg.hash_scale, cfg.stack_ring) != (0, 0, 16):
        assert layout(**pick) != layout(), pick

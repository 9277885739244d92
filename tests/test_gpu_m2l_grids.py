"""M2L (orders 1..6) where two launches differ on both trees: a warp a sink up to 304 blocks
of four, four sinks a warp beyond, at most tile_m2l_blocks blocks an SM.  Above 608 nodes
tile_m2l_blocks = 1 (152 blocks) gives a warp other sinks before than 64 does: the same bits."""
import numpy as np
import pytest

from paper_2006_14952_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tree", [0, 1])
@pytest.mark.parametrize("order", [1, 4, 5, 6])
def test_locals_do_not_depend_on_the_grid(tree, order):
    import torch

    from paper_2006_14952_gb300 import hfmm

    pos, mass = W.nfw_clustered(2500, 5, 0.5, 17)
    p = torch.from_numpy(np.ascontiguousarray(pos, dtype=np.float64)).cuda()
    m = torch.from_numpy(np.ascontiguousarray(mass, dtype=np.float32)).cuda()
    out = []
    for blocks in (0, 1, 64):
        s = hfmm.Solver(tree=tree, order=order, theta=0.9, leaf_max=8, tile_m2l_blocks=blocks)
        s.build_tree(p, m)
        s.short_range_forces()
        torch.cuda.synchronize()
        st = s.get_stats()
        assert 608 < st["nnodes"] < 4 * 304 * 4 and st["nm2l"] > 0
        out.append(s.export("locals"))
    np.testing.assert_array_equal(out[0], out[1])
    np.testing.assert_array_equal(out[0], out[2])

"""M2L's look-ahead over batches and sinks (orders 1..6): a sink's local expansion does not
depend on which sinks its warp took before it, so one block per SM (many sinks a warp, the
copies of one sink under another's arithmetic) and the most blocks allowed (one or none)
give the same bits, in either tree, for list lengths around a batch of 32."""
import numpy as np
import pytest

from paper_2006_14952_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tree", [0, 1])
@pytest.mark.parametrize("order", [1, 2, 3, 4, 5, 6])
@pytest.mark.parametrize("n,theta", [(1500, 0.9), (30011, 0.5)])
def test_locals_do_not_depend_on_the_blocks(tree, order, n, theta):
    import torch

    from paper_2006_14952_gb300 import hfmm

    pos, mass = W.nfw_clustered(n, 20, 0.5, 5)
    p = torch.from_numpy(np.ascontiguousarray(pos, dtype=np.float64)).cuda()
    m = torch.from_numpy(np.ascontiguousarray(mass, dtype=np.float32)).cuda()
    out = []
    for blocks in (1, 64):
        s = hfmm.Solver(tree=tree, order=order, theta=theta, leaf_max=8, tile_m2l_blocks=blocks)
        s.build_tree(p, m)
        acc = s.short_range_forces()
        torch.cuda.synchronize()
        assert s.get_stats()["nm2l"] > 0
        out.append((s.export("locals"), acc.cpu().numpy()))
    np.testing.assert_array_equal(out[0][0], out[1][0])
    np.testing.assert_array_equal(out[0][1], out[1][1])

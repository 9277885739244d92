"""The octree build's two tile sizes: 256 particles up to 155,648 of them (152 x 1024), 1024
beyond, at the edges of the tiles and on both sides of the change.  Nodes bit-exact against
the oracle's."""
import numpy as np
import pytest

from test_gpu_parity import run_oracle, solver
from test_gpu_tree_edges import _set

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["uniform", "clumps"])
@pytest.mark.parametrize("n,leaf", [(255, 1), (256, 16), (257, 64), (513, 3), (4096, 16), (155647, 48), (155648, 16),
                                    (155649, 16), (156673, 64), (200000, 1)])
def test_nodes_at_tile_edges(n, leaf, kind):
    import torch

    pos, mass = _set(n, kind)
    s = solver(leaf_max=leaf, order=2)
    s.build_tree(torch.from_numpy(np.ascontiguousarray(pos)).cuda(), torch.from_numpy(mass).cuda())
    f = run_oracle(pos, mass, s)
    nodes = s.export("nodes")
    np.testing.assert_array_equal(nodes, f.nodes())
    key, perm, _ = f.particles()
    np.testing.assert_array_equal(s.export("perm").astype(np.int64), perm)
    st = s.get_stats()
    assert st["nleaves"] == (nodes[:, 6] < 0).sum() and st["nlevels"] == nodes[:, 0].max() + 1

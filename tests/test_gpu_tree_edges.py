"""The octree from the sorted keys at the edges of its 1024-particle tiles and of
the leaf limit: runs of equal keys longer than a leaf (leaves at the depth cap),
cells that split across a tile's end, a root that is a leaf.  Nodes bit-exact
against the oracle's; leaves in node order; offsets from the leaf centre."""
import numpy as np
import pytest

from paper_2006_14952_gb300 import workloads as W
from test_gpu_parity import run_oracle, solver

pytestmark = pytest.mark.gpu


def _set(n, kind):
    pos, mass = W.uniform(n, n + 5)
    if kind == "clumps":  # a third of the particles on a few points, a third in tight pairs of cells
        rng = np.random.default_rng(n)
        k = n // 3
        pos[:, :k] = rng.random((3, 4))[:, rng.integers(0, 4, k)]
        pos[:, k:2 * k] = 0.5 + rng.integers(-2, 2, (3, k)) * 2.0 ** -21
    return pos, mass


@pytest.mark.parametrize("n", [1, 2, 64, 65, 1023, 1024, 1025, 3001])
@pytest.mark.parametrize("leaf", [1, 16, 64])
@pytest.mark.parametrize("kind", ["uniform", "clumps"])
def test_nodes_at_tile_and_leaf_edges(n, leaf, kind):
    import torch

    pos, mass = _set(n, kind)
    s = solver(leaf_max=leaf, order=2)
    s.build_tree(torch.from_numpy(np.ascontiguousarray(pos)).cuda(), torch.from_numpy(mass).cuda())
    f = run_oracle(pos, mass, s)
    nodes = s.export("nodes")
    np.testing.assert_array_equal(nodes, f.nodes())
    st = s.get_stats()
    assert st["nleaves"] == (nodes[:, 6] < 0).sum() and st["nlevels"] == nodes[:, 0].max() + 1

"""The tree builds' bounded waits giving up: a sort tile, or a partition tile of the k-d
build, that does not wait for its predecessors' counts takes them from the keys or the
flags.  wait_polls = -1 makes every tile do so, 1 some of them: the same nodes and the
same permutation, bit for bit."""
import numpy as np
import pytest

from paper_2006_14952_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def build(pos, mass, **kw):
    import torch

    from paper_2006_14952_gb300 import hfmm

    s = hfmm.Solver(**kw)
    s.build_tree(torch.from_numpy(np.ascontiguousarray(pos, dtype=np.float64)).cuda(),
                 torch.from_numpy(np.ascontiguousarray(mass, dtype=np.float32)).cuda())
    return s


# 2048- and 4096-key tiles of the sort, 2048-particle tiles of the partition: full and ragged
@pytest.mark.parametrize("polls", [-1, 1])
@pytest.mark.parametrize("n", [8193, 40960, 100_003, 1_100_001])
@pytest.mark.parametrize("tree", [0, 1])
def test_the_same_tree(tree, n, polls):
    pos, mass = W.nfw_clustered(n, max(1, n // 1000), 0.7, 13)
    pos[:, 5:n:7] = pos[:, 0:n - 5:7]  # equal keys: the order of the input decides
    a, b = (build(pos, mass, tree=tree, leaf_max=24, wait_polls=p) for p in (0, polls))
    for what in ("perm", "nodes") if tree == 0 else ("perm", "kd_nodes", "kd_boxes"):
        np.testing.assert_array_equal(a.export(what), b.export(what))

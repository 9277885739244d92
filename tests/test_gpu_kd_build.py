"""The k-d tree's build at the edges of its kernels: nodes of 2048 particles (one block
takes a node to its leaves), tiles of 2048 of the level partition, last levels that split
in part, one-particle leaves, and coordinates with ties.  Exact: nodes, boxes and
particle order are the oracle's."""
import numpy as np
import pytest

import oracle
from paper_2006_14952_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ties", [False, True])
@pytest.mark.parametrize(
    "n,leaf",
    [(2, 1), (3, 2), (16, 16), (17, 16), (33, 16), (1000, 1), (2047, 1), (2048, 16), (2049, 16), (4096, 1), (4097, 64),
     (8193, 5), (16385, 2), (65536, 16), (65537, 16), (100003, 3), (131071, 64), (300001, 37)])
def test_build_bit_exact(n, leaf, ties):
    import torch

    from paper_2006_14952_gb300 import hfmm

    pos, mass = W.uniform(n, 3 + n)
    if ties:  # 64 distinct values a coordinate; every eighth particle on one point
        pos = np.floor(np.asarray(pos) * 64.0) / 64.0
        flat = pos.reshape(-1)
        assert flat.size == 3 * n
        p3 = pos.reshape(3, n) if pos.shape[0] == 3 else pos.T
        p3[:, ::8] = 0.25
    s = hfmm.Solver(tree=1, leaf_max=leaf)
    s.build_tree(torch.from_numpy(np.ascontiguousarray(pos, dtype=np.float64)).cuda(),
                 torch.from_numpy(np.ascontiguousarray(mass, dtype=np.float32)).cuda())
    p = s.params
    f = oracle.KdFMM(box=p.box, rs=s.rs, rc=s.rc, G=p.G, theta=p.theta, order=p.order, leaf_max=leaf)
    f.build_tree(pos, np.asarray(mass, dtype=np.float32).astype(np.float64))
    nodes, boxes, perm = f.tree()
    np.testing.assert_array_equal(s.export("kd_nodes"), nodes)
    np.testing.assert_array_equal(s.export("kd_boxes"), boxes)
    np.testing.assert_array_equal(s.export("perm").astype(np.int64), perm)
    st = s.get_stats()
    assert st["nnodes"] == len(nodes) and st["nlevels"] == f.size("levels")
    assert st["nleaves"] == int((nodes[:, 3] < 0).sum())

"""Training pairs are collected once each, however often the walk is repeated with grown
lists: the same set from a context whose lists overflow as from one whose lists fit."""
import numpy as np
import pytest

from paper_2006_14952_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_candidates_are_collected_once():
    import torch

    from paper_2006_14952_gb300 import hfmm

    pos, mass = W.nfw_clustered(6001, 6, 0.7, 11)
    pos = torch.from_numpy(np.ascontiguousarray(pos, dtype=np.float64)).cuda()
    mass = torch.from_numpy(np.ascontiguousarray(mass, dtype=np.float32)).cuda()
    rows = {}
    for init in (1, 50_000_000):
        s = hfmm.Solver(order=8, leaf_max=32, list_init=init)
        s.build_tree(pos, mass)
        feat, err = s.collect_training_pairs(2_000_000, 3)
        assert (s.get_stats()["traverse_walks"] > 1) == (init == 1)
        r = s.export("candidates")
        assert len(r) == len(feat) and 100 < len(r) < 2_000_000
        rows[init] = r[np.lexsort((r[:, 2], r[:, 1], r[:, 0]))]
    assert len(np.unique(rows[1], axis=0)) == len(rows[1])
    np.testing.assert_array_equal(rows[1], rows[50_000_000])

"""The k-d walk's sessions shared by a group of warps (levels with fewer nodes than warps:
eight, four or two warps a node), also where a warp's part outgrows what shared memory
stages: wide cut-offs, small angles, the conventional walk.  Exact: the lists are the
oracle's as sets, each sink's entries once; the same forces, bit for bit, on a second call."""
import numpy as np
import pytest

import oracle
from paper_2006_14952_gb300 import workloads as W
from test_gpu_kd_walk import rows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,leaf,theta", [(2, 1, 0.5), (9, 1, 0.5), (130, 2, 0.3), (600, 1, 0.0), (1023, 2, 0.4),
                                          (2500, 2, 0.02), (8200, 2, 0.02)])
def test_lists_are_the_oracles(n, leaf, theta):
    import torch

    from paper_2006_14952_gb300 import hfmm

    pos, mass = W.nfw_clustered(n, 3, 0.4, 19) if n > 1000 else W.uniform(n, 19)
    s = hfmm.Solver(tree=1, pm_grid=12, theta=theta, leaf_max=leaf, order=2)
    s.build_tree(torch.from_numpy(np.ascontiguousarray(pos, dtype=np.float64)).cuda(),
                 torch.from_numpy(np.ascontiguousarray(mass, dtype=np.float32)).cuda())
    acc = s.short_range_forces().clone()
    torch.cuda.synchronize()
    p = s.params
    f = oracle.KdFMM(box=p.box, rs=s.rs, rc=s.rc, G=p.G, theta=p.theta, order=p.order, leaf_max=leaf,
                     transition_rule=p.transition_rule, size_rule=p.size_rule)
    f.build_tree(pos, np.asarray(mass, dtype=np.float32).astype(np.float64))
    f.traverse()
    p2p, m2l = f.lists()
    np.testing.assert_array_equal(rows(s.export("p2p")), rows(p2p))
    np.testing.assert_array_equal(rows(s.export("m2l")), rows(m2l))
    again = s.short_range_forces()
    torch.cuda.synchronize()
    assert torch.equal(acc, again)


@pytest.mark.parametrize("conventional", [False, True])
@pytest.mark.parametrize("n,leaf,theta", [(50, 1, 0.3), (3000, 4, 0.1), (20011, 16, 0.5)])
def test_counts_are_the_oracles(n, leaf, theta, conventional):
    import torch

    from paper_2006_14952_gb300 import hfmm

    pos, mass = W.nfw_clustered(n, 3, 0.4, 23) if n > 1000 else W.uniform(n, 23)
    s = hfmm.Solver(tree=1, pm_grid=16, theta=theta, leaf_max=leaf, order=2, list_init=7)
    s.build_tree(torch.from_numpy(np.ascontiguousarray(pos, dtype=np.float64)).cuda(),
                 torch.from_numpy(np.ascontiguousarray(mass, dtype=np.float32)).cuda())
    p = s.params
    f = oracle.KdFMM(box=p.box, rs=s.rs, rc=s.rc, G=p.G, theta=p.theta, order=p.order, leaf_max=leaf,
                     transition_rule=p.transition_rule, size_rule=p.size_rule)
    f.build_tree(pos, np.asarray(mass, dtype=np.float32).astype(np.float64))
    got = s.interaction_counts(conventional=conventional)
    f.traverse(conventional=conventional)
    want = f.counts()
    assert got["m2l"] == want["m2l"] and got["p2p"] == want["p2p"]
    assert got["p2p_particle_pairs"] == want["p2p_particle_pairs"]

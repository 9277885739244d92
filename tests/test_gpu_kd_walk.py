"""The k-d walk's sessions beyond what shared memory stages (1024 entries a sink: counted, then
written by a second walk of the sink), with one-particle leaves and a cut-off of a third of
the box, small angles and both size rules.  Exact: the lists are the oracle's as sets, each
sink's entries once; the same lists again on a second call, and forces with the same bits."""
import numpy as np
import pytest

import oracle
from paper_2006_14952_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def rows(a):
    a = np.asarray(a, dtype=np.int64).reshape(-1, 3)
    return a[np.lexsort((a[:, 2], a[:, 1], a[:, 0]))]


@pytest.mark.parametrize("size_rule", [0, 1])
@pytest.mark.parametrize("n,leaf,theta,longest", [(7000, 1, 0.15, 1), (9000, 2, 0.2, 1025), (1, 1, 0.5, 1),
                                                  (40, 8, 0.5, 27), (3000, 7, 0.9, 200)])
def test_lists_are_the_oracles(n, leaf, theta, longest, size_rule):
    import torch

    from paper_2006_14952_gb300 import hfmm

    pos, mass = W.uniform(n, 17)
    s = hfmm.Solver(tree=1, pm_grid=17, theta=theta, leaf_max=leaf, order=2, size_rule=size_rule)
    s.build_tree(torch.from_numpy(np.ascontiguousarray(pos, dtype=np.float64)).cuda(),
                 torch.from_numpy(np.ascontiguousarray(mass, dtype=np.float32)).cuda())
    acc = s.short_range_forces().clone()
    torch.cuda.synchronize()
    p = s.params
    f = oracle.KdFMM(box=p.box, rs=s.rs, rc=s.rc, G=p.G, theta=p.theta, order=p.order, leaf_max=leaf,
                     transition_rule=p.transition_rule, size_rule=size_rule)
    f.build_tree(pos, np.asarray(mass, dtype=np.float32).astype(np.float64))
    f.traverse()
    p2p, m2l = f.lists()
    np.testing.assert_array_equal(rows(s.export("p2p")), rows(p2p))
    np.testing.assert_array_equal(rows(s.export("m2l")), rows(m2l))
    assert np.bincount(rows(p2p)[:, 0]).max() >= longest
    again = s.short_range_forces()
    torch.cuda.synchronize()
    assert torch.equal(acc, again)

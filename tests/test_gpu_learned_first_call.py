"""Weights loaded just before the first learned walk, on a stream that waits for no
other: the same bits as in a later call show that they were there before the walk."""
import os

import numpy as np
import pytest

from paper_2006_14952_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_first_learned_call_on_a_side_stream():
    import torch

    import paper_2006_14952_gb300 as package
    from paper_2006_14952_gb300 import hfmm

    weights = np.fromfile(os.path.join(os.path.dirname(package.__file__), "weights", "mac_weights.bin"), np.uint16)
    pos, mass = W.nfw_clustered(20011, 20, 0.7, 6)
    pos = torch.from_numpy(np.ascontiguousarray(pos, dtype=np.float64)).cuda()
    mass = torch.from_numpy(np.ascontiguousarray(mass, dtype=np.float32)).cuda()
    s = hfmm.Solver(pm_grid=32, mac_mode=1, order=6, leaf_max=48)
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.Stream()):
        s.build_tree(pos, mass)
        s.load_mlp(weights)
        first = s.short_range_forces()
        again = s.short_range_forces()
        torch.cuda.current_stream().synchronize()
    assert torch.isfinite(first).all() and torch.equal(first, again)

"""The mesh call as a context's first call on a stream that waits for no other: its
tables are uploaded in that call, so the same bits as in later calls show that they
were there before their readers."""
import numpy as np
import pytest

from paper_2006_14952_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("split", [0, 1])
@pytest.mark.parametrize("ng", [33, 64])
def test_first_call_on_a_side_stream(split, ng):
    import torch

    from paper_2006_14952_gb300 import hfmm

    pos, mass = W.nfw_clustered(20011, 20, 0.7, 5)
    pos = torch.from_numpy(np.ascontiguousarray(pos, dtype=np.float64)).cuda()
    mass = torch.from_numpy(np.ascontiguousarray(mass, dtype=np.float32)).cuda()
    zero = torch.zeros(3, 20011, device="cuda")
    s = hfmm.Solver(pm_grid=ng, split=split)
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        s.build_tree(pos, mass)
        first = s.pm_long_range(zero.clone())
        again = s.pm_long_range(zero.clone())
    side.synchronize()
    later = s.pm_long_range(zero.clone())
    assert torch.isfinite(first).all() and first.abs().max() > 0
    assert torch.equal(first, again) and torch.equal(first, later)

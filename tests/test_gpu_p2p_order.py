"""P2P with its work ordered (512 leaves or more) and taken as it comes (fewer), in one batch
and in sink batches (where most leaves' lists are empty): theta 0, all pairs by P2P, against
the FP64 direct sum within the 1e-5 relative RMS of the other theta-0 tests."""
import numpy as np
import pytest

import oracle
from paper_2006_14952_gb300 import workloads as W
from test_gpu_parity import run_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batches", [1, 3])
@pytest.mark.parametrize("n,leaf,fewer", [(700, 64, True), (3000, 16, None), (3000, 64, True), (4000, 2, False),
                                          (511, 1, None)])
def test_theta_zero_equals_direct_sum(n, leaf, fewer, batches):
    pos, mass = W.uniform(n, 23)
    s, acc = run_gpu(pos, mass, pm_grid=24, theta=0.0, leaf_max=leaf, sink_batches=batches)
    st = s.get_stats()
    if fewer is not None:
        assert (st["nleaves"] < 512) == fewer
    ref = oracle.direct_sr(pos, mass, 1.0, s.rs, s.rc)
    assert np.sqrt(((acc - ref) ** 2).sum() / (ref ** 2).sum()) < 1e-5

"""Leaves of more than 64 particles: a cell on the deepest level holds however many
coincide in it.  theta 0, all pairs by P2P, below and above the 512 leaves from which
the work is ordered (and such a leaf's shared by a block), in one batch and in several,
against the FP64 direct sum: 1e-5 relative RMS as in the other theta-0 tests, over the
crowded particles alone too (coincident pairs have no force)."""
import numpy as np
import pytest

import oracle
from paper_2006_14952_gb300 import workloads as W
from test_gpu_parity import run_gpu

pytestmark = pytest.mark.gpu


def crowded(n, crowd, seed):
    """n uniform particles, 2 `crowd` of them moved to two points, in input order at random.
    (Mutual P2P: of two leaves the deeper one owns a pair, so only two such leaves react.)"""
    rng = np.random.default_rng(seed)
    pos, mass = W.uniform(n, seed)
    pos[:, :crowd] = np.array([0.3137, 0.7071, 0.5772])[:, None]
    pos[:, crowd:2 * crowd] = np.array([0.4142, 0.6931, 0.6180])[:, None]
    order = rng.permutation(n)
    return np.ascontiguousarray(pos[:, order]), mass, order < 2 * crowd


@pytest.mark.parametrize("opts", [{}, {"sink_batches": 3}, {"split": 1}, {"p2p_mutual": 1}],
                         ids=["plain", "batches", "poly", "mutual"])
@pytest.mark.parametrize("n", [700, 12000])
@pytest.mark.parametrize("crowd", [65, 96, 100, 300])
def test_theta_zero_equals_direct_sum(crowd, n, opts):
    pos, mass, is_crowd = crowded(n + 2 * crowd, crowd, 31 + crowd)
    s, acc = run_gpu(pos, mass, pm_grid=24, theta=0.0, leaf_max=16, **opts)
    assert (s.get_stats()["nleaves"] < 512) == (n == 700)
    nodes = s.export("nodes")
    assert (nodes[nodes[:, 6] < 0, 5] == crowd).sum() == 2
    ref = oracle.direct_sr(pos, mass, 1.0, s.rs, s.rc, **({"split": "poly"} if opts.get("split") else {}))
    for which in (slice(None), is_crowd):
        a, r = acc[:, which], ref[:, which]
        assert np.sqrt(((a - r) ** 2).sum() / (r ** 2).sum()) < 1e-5

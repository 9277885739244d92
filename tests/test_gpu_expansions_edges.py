"""The upward and downward passes at the edges of their kernels: trees of one to five and
more levels (the first three with children go through one block), leaves of one particle,
of fewer than the lanes that share a leaf, and of 64.  Multipoles and locals of every cell
against the FP64 oracle on the same tree, by degree: FP32 sums of at most 64 particles, 8
children a level and some hundred translated terms of either sign, all O(1) in the scaled
form: 1e-5 relative per degree over all cells, the bound of the expansions' parity test."""
import numpy as np
import pytest

import oracle
from paper_2006_14952_gb300 import workloads as W
from test_gpu_parity import run_gpu, run_oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [1, 4, 6])
@pytest.mark.parametrize("n,leaf,levels", [(1, 1, 1), (64, 64, 1), (65, 64, 2), (9, 1, 2), (200, 3, 3), (1000, 2, 5),
                                           (5000, 16, 5), (40000, 63, 5)])
def test_expansions_by_degree(n, leaf, levels, order):
    pos, mass = W.nfw_clustered(n, 5, 0.3, 4) if n >= 5000 else W.uniform(n, 6)
    s, _ = run_gpu(pos, mass, pm_grid=32, theta=0.7, order=order, leaf_max=leaf)
    assert s.get_stats()["nlevels"] >= levels
    f = run_oracle(pos, mass, s)
    f.forces()
    nodes = s.export("nodes")
    h = 1.0 / 2.0 ** nodes[:, 0]
    deg = oracle.multi_indices(order).sum(axis=1)
    Mg = s.export("multipoles").astype(np.float64) * h[:, None] ** deg[None, :]
    Lg = s.export("locals").astype(np.float64) / h[:, None] ** (deg[None, :] + 1)
    for g, o in ((Mg, f.expansions("M")), (Lg, f.expansions("L"))):
        for k in range(order + 1):
            sel = deg == k
            err = np.sqrt(((g[:, sel] - o[:, sel]) ** 2).sum() / max((o[:, sel] ** 2).sum(), 1e-300))
            assert err < 1e-5, (k, err)

"""The sink-driven walk where its sessions change shape: a root that is a leaf,
sessions whose entries outgrow the stage in shared memory (walked twice), leaves
beside much denser regions (many nodes waiting on the stack), deep trees, and
few or many blocks.  The lists have to equal the oracle's, and the pairs
classified those of the oracle's walk."""
import numpy as np
import pytest

from paper_2006_14952_gb300 import workloads as W
from test_gpu_parity import run_gpu, run_oracle, sorted_rows

pytestmark = pytest.mark.gpu


def _spike(n, width, seed):
    """Half the particles uniform, half in one tight clump: large leaves beside tiny ones."""
    pos, mass = W.uniform(n, seed)
    rng = np.random.default_rng(seed + 1)
    pos[:, : n // 2] = np.mod(0.37 + width * rng.standard_normal((3, n // 2)), 1.0)
    return pos, mass


@pytest.mark.parametrize("name,kw", [
    ("root-leaf", dict(leaf_max=64)),
    ("one-level", dict(leaf_max=16)),
    ("leaf-one", dict(leaf_max=1, theta=0.5, order=2)),
    ("spike", dict(leaf_max=4, theta=0.3, order=2)),
    ("spike-tight", dict(leaf_max=8, theta=0.6, order=3, size_rule=0, transition_rule=0)),
    ("wide-cutoff", dict(leaf_max=2, theta=0.2, order=2, pm_grid=12)),
])
def test_lists_where_sessions_change_shape(name, kw):
    pos, mass = {"root-leaf": lambda: W.uniform(64, 301), "one-level": lambda: W.uniform(65, 302),
                 "leaf-one": lambda: W.nfw_clustered(6000, 2, 0.9, 303), "spike": lambda: _spike(20000, 3e-3, 304),
                 "spike-tight": lambda: _spike(30000, 1e-5, 305),
                 "wide-cutoff": lambda: W.uniform(5000, 306)}[name]()
    kw = dict(dict(pm_grid=32, order=4, theta=0.5), **kw)
    s, _ = run_gpu(pos, mass, **kw)
    f = run_oracle(pos, mass, s)
    f.traverse()
    p2p, m2l = f.lists()
    np.testing.assert_array_equal(sorted_rows(s.export("p2p")), sorted_rows(p2p))
    np.testing.assert_array_equal(sorted_rows(s.export("m2l")), sorted_rows(m2l))
    counts = s.interaction_counts()
    assert counts["p2p"] == len(p2p) and counts["m2l"] == len(m2l)
    assert counts["frontier_pairs"] == s.get_stats()["frontier_pairs"]

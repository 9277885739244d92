"""The octree walk's bounded wait giving up: an error status that says so, the same from
every call that walks, and a context that still works; also when a list overflows in the
same walk (which alone would repeat it with grown lists)."""
import ctypes

import numpy as np
import pytest

from paper_2006_14952_gb300 import workloads as W


def test_wait_polls_is_checked():
    from paper_2006_14952_gb300 import hfmm

    L = hfmm.load()
    p, h = hfmm.default_params(), ctypes.c_void_p()
    assert p.wait_polls == 0
    p.wait_polls = -2
    assert L.hfmm_create(ctypes.byref(p), ctypes.byref(h)) == -1 and b"wait_polls" in L.hfmm_last_error(None)


def particles(n=20011):
    import torch

    pos, mass = W.nfw_clustered(n, 20, 0.7, 7)
    return (torch.from_numpy(np.ascontiguousarray(pos, dtype=np.float64)).cuda(),
            torch.from_numpy(np.ascontiguousarray(mass, dtype=np.float32)).cuda())


def good(pos, mass):
    from paper_2006_14952_gb300 import hfmm

    s = hfmm.Solver()
    s.build_tree(pos, mass)
    return s.short_range_forces()


@pytest.mark.gpu
@pytest.mark.parametrize("opts", [{}, {"sink_batches": 3}, {"use_graph": 1}, {"p2p_mutual": 1}],
                         ids=["direct", "batches", "graph", "mutual"])
def test_a_wait_that_gives_up_is_a_timeout(opts):
    import torch

    from paper_2006_14952_gb300 import hfmm

    pos, mass = particles()
    s = hfmm.Solver(wait_polls=-1, **opts)
    s.build_tree(pos, mass)
    for call in (s.short_range_forces, s.interaction_counts):
        with pytest.raises(hfmm.HfmmError, match="HFMM_ERR_TIMEOUT"):
            call()
    vel, acc = torch.zeros(3, pos.shape[1], device="cuda"), torch.zeros(3, pos.shape[1], device="cuda")
    with pytest.raises(hfmm.HfmmError, match="HFMM_ERR_TIMEOUT"):
        s.step(pos.clone(), vel, acc, 1e-4)
    assert torch.equal(good(pos, mass), good(pos, mass))


@pytest.mark.gpu
def test_an_overflowing_list_does_not_hide_it():
    """One poll finds the root, whose open list of one entry overflows well after the other blocks gave up."""
    from paper_2006_14952_gb300 import hfmm

    pos, mass = particles()
    s = hfmm.Solver(wait_polls=1, list_init=1)
    s.build_tree(pos, mass)
    with pytest.raises(hfmm.HfmmError, match="HFMM_ERR_TIMEOUT"):
        s.short_range_forces()

"""A label outside 0..7 has no class weight: beside class weights such a sample counts as
one of weight zero, and nothing is read outside the eight weights."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_labels_without_a_class_weight():
    import torch

    from paper_2006_14952_gb300 import hfmm

    rng = np.random.default_rng(3)
    n = 1000
    w = torch.tensor(0.3 * rng.standard_normal(hfmm.MLP_WEIGHTS), dtype=torch.float32).cuda()
    x = torch.tensor(rng.uniform(-1, 1, (n, 12)), dtype=torch.float32).cuda()
    cw = torch.tensor(list(rng.uniform(0.5, 2.0, 7)) + [0.0], dtype=torch.float32).cuda()
    y = torch.tensor(rng.integers(0, 7, n), dtype=torch.int32).cuda()
    out, zero = y.clone(), y.clone()
    out[::10] = torch.tensor([-1, 8, 1 << 30, -(1 << 31)] * 25, dtype=torch.int64).to(torch.int32).cuda()
    zero[::10] = 7
    s = hfmm.Solver()
    for a, b in zip(s.mlp_grad(w, x, out, cw), s.mlp_grad(w, x, zero, cw)):
        assert torch.isfinite(a).all() and torch.equal(a, b)

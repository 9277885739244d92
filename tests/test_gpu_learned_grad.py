"""Training gradients at the edges of the gradient kernel's 64-sample tiles and
of its grid, against the oracle's backward.

Inputs, weights and biases are small multiples of powers of two, so every
pre-activation is exact in FP32 in any order of summation and the BF16
activations cannot differ from the oracle's; the label of a sample is never its
most likely class, so no gradient is a small difference of large numbers.  What
remains is FP32 rounding of the softmax (about 2^-20 relative) and of sums of n
terms: 1e-5 of the gradient's norm, and 1e-4 of |g| + 1e-2 rms(g) per element.
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def exact_network(seed):
    rng = np.random.default_rng(seed)
    w = rng.integers(-4, 5, 5512) / 8.0
    w[832 + 4096 + 64:832 + 4096 + 64 + 512] /= 8.0
    return w


@pytest.mark.parametrize("n", [1, 15, 64, 65, 29183, 29185])
def test_gradient_at_tile_edges(n):
    import torch

    from paper_2006_14952_gb300 import hfmm

    w = exact_network(n)
    rng = np.random.default_rng(n + 1)
    x = rng.integers(-8, 9, (n, 12)) / 4.0
    y = ((oracle.mlp_forward(w, x).argmax(axis=1) + rng.integers(1, 8, n)) % 8).astype(np.int32)
    cw = rng.uniform(0.5, 2.0, 8).astype(np.float32)
    s = hfmm.Solver()
    args = (torch.tensor(w, dtype=torch.float32).cuda(), torch.tensor(x, dtype=torch.float32).cuda(),
            torch.tensor(y).cuda(), torch.tensor(cw).cuda())
    g, loss = s.mlp_grad(*args)
    g2, loss2 = s.mlp_grad(*args)
    assert torch.equal(g, g2) and torch.equal(loss, loss2)  # no atomics: the same bits on every run
    ref_loss, ref = oracle.mlp_loss_grad(w, x, y, cw.astype(np.float64), rnd=1)
    dev = np.abs(g.cpu().numpy().astype(np.float64) - ref)
    assert loss.item() == pytest.approx(ref_loss, rel=1e-5)
    assert np.linalg.norm(dev) < 1e-5 * np.linalg.norm(ref)
    assert np.all(dev <= 1e-4 * (np.abs(ref) + 1e-2 * np.sqrt((ref ** 2).mean())))


def test_a_nan_feature_stays_out_of_the_weight_gradients():
    """A NaN input makes every first-layer unit of its sample inactive: its terms are left out, not added as NaN."""
    import torch

    from paper_2006_14952_gb300 import hfmm

    w = exact_network(3)
    x = np.random.default_rng(4).integers(-8, 9, (70, 12)) / 4.0
    x[66, 5] = np.nan
    g, loss = hfmm.Solver().mlp_grad(torch.tensor(w, dtype=torch.float32).cuda(),
                                     torch.tensor(x, dtype=torch.float32).cuda(),
                                     torch.arange(70, dtype=torch.int32).remainder(8).cuda())
    assert torch.isfinite(g).all() and torch.isfinite(loss).all()

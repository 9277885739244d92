"""The training gradient where a forward sum decides a rounding: the samples of a
random batch with a first-layer sum so close to a BF16 rounding boundary that the
order and the rounding of the additions decide the activation, and with it the
sign of second-layer sums near zero.

Reference: the forward pass in FP32 FMAs, the bias first and the inputs in order
(BF16 products are exact in FP32, so an FMA is an FP32 addition of the product),
the backward pass in FP64 on its activations.  What remains is the softmax in FP32
(2^-20 relative) and some twenty BF16 roundings of second-layer activations among
a million (up to 3e-7 together): 2e-6 of the gradient's norm.  Where sums are
truncated instead, a ReLU gate of a sample flips in five of these twelve batches:
1e-5 and more.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

POOL = 400_000


def pool(seed):
    """Features, labels and a fresh network of the training case's kind."""
    rng = np.random.default_rng(seed)
    sc, ha, hb = rng.uniform(0.1, 4.0, POOL), rng.uniform(0.05, 0.5, POOL), rng.uniform(0.05, 0.5, POOL)
    x = np.stack([sc, 0.6 * sc, 0.3 * sc, ha, hb, np.maximum(ha, hb), rng.integers(-2, 3, POOL) / 8.0,
                  rng.uniform(0.1, 1.0, POOL), rng.uniform(0.1, 1.0, POOL), 0.2 * abs(rng.standard_normal(POOL)),
                  0.1 * abs(rng.standard_normal(POOL)), sc / 4.5], axis=1).astype(np.float32)
    w = [((2.0 / a) ** 0.5 * rng.standard_normal((b, a)), 0.05 * rng.standard_normal(b))
         for a, b in ((12, 64), (64, 64), (64, 8))]
    return x, rng.integers(0, 8, POOL).astype(np.int32), rng.uniform(0.5, 2.0, 8).astype(np.float32), w


def bf16(t):
    import torch
    return t.to(torch.bfloat16).to(t.dtype)


def fma_layer(h, w, b):
    z = b[None, :].expand(h.shape[0], -1)
    for k in range(w.shape[1]):
        z = z + h[:, k:k + 1] * w[None, :, k]
    return z


def near_a_boundary(x, w, b):
    """Rows with a positive sum within 2^-22 of its terms from a BF16 rounding boundary."""
    import torch
    z = x.double() @ w.double().T + b.double()
    terms = x.double().abs() @ w.double().abs().T + b.double().abs()
    mant, exp = torch.frexp(z)
    unit = torch.ldexp(torch.ones_like(z), exp - 8)  # of a BF16 value like z
    off = (mant * 256 - torch.floor(mant * 256) - 0.5).abs() * unit
    return ((off < terms * 2.0 ** -22) & (z > 0)).any(1)


def reference(x, y, cw, w):
    import torch
    z1 = fma_layer(x, *w[0])
    h1 = bf16(z1.clamp(min=0))
    z2 = fma_layer(h1, *w[1])
    h2 = bf16(z2.clamp(min=0))
    p = torch.softmax(fma_layer(h2, *w[2]).double(), 1)
    d3 = p.clone()
    d3[torch.arange(len(y)), y.long()] -= 1.0
    d3 *= cw.double()[y.long()][:, None]
    d2 = (d3 @ w[2][0].double()) * (z2 > 0)
    d1 = (d2 @ w[1][0].double()) * (z1 > 0)
    return torch.cat([t.reshape(-1) for t in (d1.T @ x.double(), d1.sum(0), d2.T @ h1.double(), d2.sum(0),
                                              d3.T @ h2.double(), d3.sum(0))]) / len(y)


@pytest.mark.parametrize("seed", range(12))
def test_gradient_with_sums_at_rounding_boundaries(seed):
    import torch

    from paper_2006_14952_gb300 import hfmm

    x, y, cw, w = pool(seed)
    x, y, cw = (torch.tensor(v).cuda() for v in (x, y, cw))
    flat = torch.cat([torch.tensor(v, dtype=torch.float32).reshape(-1) for layer in w for v in layer]).cuda()
    wr = [tuple(bf16(torch.tensor(v, dtype=torch.float32)).cuda() for v in layer) for layer in w]
    xr = bf16(x)
    rows = near_a_boundary(xr, *wr[0])
    assert 4000 < int(rows.sum()) < 40000
    x, xr, y = x[rows].contiguous(), xr[rows], y[rows].contiguous()
    g, _ = hfmm.Solver().mlp_grad(flat, x, y, cw)
    ref = reference(xr, y, cw, wr)
    assert (g.double() - ref).norm() < 2e-6 * ref.norm()

"""P2P's layouts of a chunk's sinks over a warp (one, two or three sinks a lane by the chunk's
size): every size of a leaf from 1 to 64 particles, the root alone, all pairs by P2P.
Against the FP64 pair sum with the particles at least 0.1 apart: FP32 offsets within 0.5 of
the leaf's centre are off by 2^-25, 2^-24 / 0.1 of a separation, three times that in 1 / r^3,
and the pair law by some 2^-22: below 3e-6 of the sum of the pairs' magnitudes; 5e-6 asked."""
import numpy as np
import pytest

from scipy.special import erfc

pytestmark = pytest.mark.gpu


def pair_sum(pos, mass, rs, rc):
    n = pos.shape[1]
    acc, mag = np.zeros((3, n)), np.zeros(n)
    for sx in (-1, 0, 1):
        for sy in (-1, 0, 1):
            for sz in (-1, 0, 1):
                d = pos[:, None, :] + np.array([sx, sy, sz], float)[:, None, None] - pos[:, :, None]  # source - sink
                r = np.sqrt((d ** 2).sum(axis=0))
                ok = (r > 0) & (r < rc)
                rr = np.where(ok, r, 1.0)
                x = rr / rs
                f = np.where(ok, mass[None, :] * (erfc(x / 2) + x * np.exp(-x * x / 4) / np.sqrt(np.pi)) / rr ** 3, 0.0)
                acc += (f[None] * d).sum(axis=2)
                mag += (f * rr).sum(axis=1)
    return acc, mag


@pytest.mark.parametrize("n", list(range(1, 65)))
@pytest.mark.parametrize("tree", [0, 1])
def test_every_chunk_size(n, tree):
    import torch

    from paper_2006_14952_gb300 import hfmm

    rng = np.random.default_rng(n)
    cells = rng.permutation(125)[:n]  # a 5^3 lattice, jittered: 0.2 - 2 x 0.05 apart at least
    grid = np.stack([cells // 25, (cells // 5) % 5, cells % 5]).astype(float)
    pos = (grid + 0.5) / 5 + rng.uniform(-0.05, 0.05, (3, n))
    mass = rng.uniform(0.5, 1.5, n).astype(np.float32) / n
    s = hfmm.Solver(tree=tree, leaf_max=64, theta=0.5, order=2, pm_grid=17)
    s.build_tree(torch.from_numpy(np.ascontiguousarray(pos)).cuda(), torch.from_numpy(mass).cuda())
    acc = s.short_range_forces()
    torch.cuda.synchronize()
    assert s.get_stats()["nm2l"] == 0
    ref, mag = pair_sum(pos, mass.astype(np.float64), s.rs, s.rc)
    err = np.abs(acc.cpu().numpy().astype(np.float64) - s.params.G * ref).max(axis=0)
    assert (err <= 5e-6 * s.params.G * mag + 1e-30).all()

"""The radix sort behind the tree build, at the edges of its single-block sizes
(1024, 2048, 4096, 8192 keys) and of its tiles (2048 keys, 4096 from 2^20 on): the sorted keys and the stable permutation, on sets
with many equal keys, so that an element out of its place or its turn shows."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 33, 1024, 1025, 2049, 4097, 8192, 8193, 10240, 70001, (1 << 20) - 1, (1 << 20) + 1, (1 << 20) + 4096 * 3])
@pytest.mark.parametrize("cells", [3, 512])
def test_sorted_keys_and_stable_permutation(n, cells):
    import torch

    from paper_2006_14952_gb300 import hfmm

    rng = np.random.default_rng(n + cells)
    pos = rng.integers(0, cells, (3, n)) / cells  # few distinct positions: long runs of equal keys
    s = hfmm.Solver(leaf_max=64)
    s.build_tree(torch.from_numpy(pos).cuda(), torch.full((n,), 1.0 / n, device="cuda"))
    keys, perm = s.export("keys"), s.export("perm")
    own = np.empty(n, np.uint64)
    own[perm] = keys
    np.testing.assert_array_equal(perm, np.argsort(own, kind="stable"))
    assert np.all(keys[1:] >= keys[:-1])
    # equal positions, and only those, have equal keys
    flat = (pos * cells).round().astype(np.int64)
    ids = (flat[0] * cells + flat[1]) * cells + flat[2]
    assert len(np.unique(own)) == len(np.unique(ids)) == len(np.unique(np.stack([own.astype(np.int64), ids]), axis=1).T)

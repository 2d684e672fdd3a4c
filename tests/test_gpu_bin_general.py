"""The integer form of the cell rule for any K / box: bit-exact against the oracle's FP64 rule on values at
and next to every cell face, halfway points, small, negative, far-away and subnormal coordinates."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def adversarial(K, box, seed):
    rng = np.random.default_rng(seed)
    w = box / K
    k = rng.integers(0, K + 1, 4000)
    faces = (k * w).astype(np.float32)
    halves = ((k + 0.5) * w).astype(np.float32)
    near = []
    for v in (faces, halves):
        for ulps in range(-3, 4):
            near.append((v.view(np.int32) + np.where(v > 0, ulps, 0).astype(np.int32)).view(np.float32))
    plain = (rng.random(60000) * box).astype(np.float32)
    small = (w * 2.0 ** rng.uniform(-75, 0, 8000)).astype(np.float32)     # t down to 2^-75: every shift of the rule
    quarter = (w * (2.0 ** -np.arange(0, 12)[:, None] + rng.uniform(-1, 1, (12, 200)) * 1e-7)).astype(np.float32).ravel()
    far = (rng.uniform(-40, 40, 4000) * box).astype(np.float32)
    huge = (rng.uniform(-1, 1, 600) * 1e12 * box).astype(np.float32)
    sub = np.array([0.0, -0.0, 1e-45, 1e-40, -1e-40, 1e-38], np.float32)
    v = np.concatenate(near + [plain, small, -small, quarter, far, huge, np.repeat(sub, 50)])
    return np.ascontiguousarray(rng.permutation(v)[: len(v) // 3 * 3].reshape(-1, 3))


@pytest.mark.parametrize("K,box", [(101, 500.0), (7, 3.7), (1, 0.3), (13, 1.3), (96, 1.0), (25, 1e-3), (11, 6.02e23),
                                   (300, 0.1), (24, 1.0 / 3.0), (64, 250.0)])
def test_bit_exact_for_any_grid_and_box(K, box):
    import torch
    import paper_2110_11392_gb300 as nf
    pos = adversarial(K, box, K)
    off, rel, perm = nf.bin_particles(torch.from_numpy(pos).cuda(), box, K)
    off_o, rel_o, perm_o = oracle.bin_particles(pos, box, K)
    assert np.array_equal(off.cpu().numpy(), off_o)
    assert np.array_equal(perm.cpu().numpy(), perm_o)
    assert np.array_equal(rel.cpu().numpy().view(np.int32), rel_o.view(np.int32))

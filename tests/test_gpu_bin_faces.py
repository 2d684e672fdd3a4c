"""nf_bin at every cell face of grids where the FP32 product K/box * x lies on the other side of the face for
some coordinates (the counting and the sorting kernel must agree there): bit-exact against the oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,box", [(32, 3.7), (64, 3.7), (128, 3.7), (31, 3.7), (34, 250.0), (68, 500.0), (109, 205.0),
                                   (101, 0.7), (183, 0.7), (155, 0.3), (212, 13.0), (8, 330.0), (127, 879.0),
                                   (75, 231.6)])
def test_faces_inside_and_outside_the_box(K, box):
    import torch
    import paper_2110_11392_gb300 as nf
    k = np.concatenate([np.arange(1, 2 * K + 1), np.unique(np.logspace(2, 6, 2000).astype(int))])
    bits = (k * (box / K)).astype(np.float32).view(np.int32)
    x = (bits[:, None] + np.arange(-4, 5, dtype=np.int32)).view(np.float32).ravel()
    x = np.concatenate([x, -x])
    rng = np.random.default_rng(K)
    pos = np.ascontiguousarray(np.stack([rng.permutation(x) for _ in range(3)], 1))
    off, rel, perm = nf.bin_particles(torch.from_numpy(pos).cuda(), box, K)
    off_o, rel_o, perm_o = oracle.bin_particles(pos, box, K)
    assert np.array_equal(off.cpu().numpy(), off_o)
    assert np.array_equal(perm.cpu().numpy(), perm_o)
    assert np.array_equal(rel.cpu().numpy().view(np.int32), rel_o.view(np.int32))

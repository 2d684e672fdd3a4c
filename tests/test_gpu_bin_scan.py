"""Count matrices at the edge of the one-block scan: at K = 8 a tile of 2048 particles has 512 counts, so 32
tiles make the largest matrix that one block scans; a reused workspace (the counters are cleared by a kernel)
gives the same results again."""
import numpy as np
import pytest

import oracle

from _helpers import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [1, 2047, 2049, 8 * 2048, 32 * 2048 - 1, 32 * 2048, 32 * 2048 + 1, 40 * 2048])
def test_bin_at_the_edges_of_the_scan(N):
    import paper_2110_11392_gb300 as nf
    pos = np.random.default_rng(N).random((N, 3)).astype(np.float32)
    off_o, rel_o, perm_o = oracle.bin_particles(pos, 1.0, 8)
    for _ in range(2):
        off, rel, perm = nf.bin_particles(to_dev(pos), 1.0, 8)
        assert np.array_equal(off.cpu().numpy(), off_o)
        assert np.array_equal(perm.cpu().numpy(), perm_o)
        assert np.array_equal(rel.cpu().numpy().view(np.int32), rel_o.view(np.int32))


def test_forces_repeat_on_one_workspace():
    import torch
    import paper_2110_11392_gb300 as nf
    from paper_2110_11392_gb300 import _lib
    pos = to_dev(np.random.default_rng(3).random((5000, 3)).astype(np.float32))
    ref = nf.forces(pos, 1.0, 6, 2, 1e-3)
    ws = torch.full((_lib.nf_workspace_bytes(5000, 6, 2),), 255, dtype=torch.uint8, device="cuda")  # nothing zero
    for _ in range(3):
        assert torch.equal(nf.forces(pos, 1.0, 6, 2, 1e-3, ws=ws), ref)

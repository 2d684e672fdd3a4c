"""The combine's one-particle-a-thread blocks and the net-force tree at the edges of a block."""
import numpy as np
import pytest

from workloads import uniform_positions

from _helpers import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [1, 255, 256, 257, 513, 65537])
def test_net_and_unaligned_output_at_block_edges(N):
    import torch
    import paper_2110_11392_gb300 as nf
    pos = to_dev(uniform_positions(N, N))
    acc, net = nf.forces(pos, 1.0, 6, 2, 1e-3, net=True)
    # FP64 sums of N terms in any order differ by at most N 2^-52 of the sum of magnitudes
    a = acc.double()
    bound = max(N, 1) * 2.0 ** -52 * a.abs().sum(0) / N
    assert bool(((net - a.sum(0) / N).abs() <= bound).all())
    # an output that starts 4 bytes past an 8-byte boundary takes the scalar stores
    buf = torch.full((3 * N + 2,), float("nan"), device="cuda")
    out = nf.forces(pos, 1.0, 6, 2, 1e-3, out=buf[1:3 * N + 1].view(N, 3))
    assert torch.equal(out, acc)
    assert np.isnan(buf[0].item()) and np.isnan(buf[-1].item())

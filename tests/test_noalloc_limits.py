"""The sizes that nf_forces_noalloc takes: its limit in particles per (K, R), and its results at the limit,
where nf_forces takes boxes of the same size through its own workspace."""
import ctypes

import pytest

from paper_2110_11392_gb300 import _lib

# the largest N per (K, R): the directed plan in chunks of 128 sinks within 32 MiB
LIMITS = [(5, 2, 268624), (20, 2, 236720), (100, 2, 60681), (60, 1, 257344), (12, 1, 308800), (3, 1, 362906),
          (9, 4, 163411), (7, 3, 212438), (64, 2, 190592)]


@pytest.mark.parametrize("K,R,N", LIMITS)
def test_limit_in_particles(K, R, N):
    fake = ctypes.c_void_p(0x7F0000001000)
    rc = _lib.load().nf_forces_noalloc(fake, N + 1, 1.0, K, R, 0.01 / K, fake, None, None)
    assert rc == _lib.NF_ERR_WORKSPACE and "needs" in _lib.nf_last_error()


@pytest.mark.gpu
@pytest.mark.parametrize("K,R,N", LIMITS)
def test_results_at_the_limit(K, R, N):
    import torch
    import paper_2110_11392_gb300 as nf
    from workloads import uniform_positions
    pos = torch.from_numpy(uniform_positions(N, K)).cuda()
    out, net = torch.empty_like(pos), torch.empty(3, dtype=torch.float64, device="cuda")
    _lib.nf_forces_noalloc(pos, 1.0, K, R, 0.01 / K, out, net)
    ref, ref_net = nf.forces(pos, 1.0, K, R, 0.01 / K, net=True)
    assert torch.equal(out, ref) and torch.equal(net, ref_net)

"""Workspace of the force calls: what the symmetric kernel's partial sums add stays bounded, so that a batch or a
wide stencil that fits the GPU with the directed kernel alone is neither refused nor too large for it."""
import pytest

from paper_2110_11392_gb300 import _lib


def batch(n, N, K, R):
    return [dict(N=N, K=K, R=R, eps=1e-4, box=1.0)] * n


def directed_bytes(N, K, R, chunk=32):
    """Lower bound of the directed plan: binning, work items and one row of partial sums a particle."""
    ns = 2 * R + 1
    return (4 + 4 + 16 + 16 + 4 + 16 + 16 * ns) * N + 16 * (ns * N // chunk + K ** 3)


def test_batch_of_many_boxes():
    n, N, K, R = 300, 10 ** 6, 25, 2
    need = _lib.nf_workspace_bytes_batched(batch(n, N, K, R))
    # 5 % for the tables per cell, the sort's counts and the work units of one lot
    assert 0 < need <= 1.05 * n * directed_bytes(N, K, R) + (8 << 30) + (1 << 30), need


def test_batch_with_many_units_is_not_refused():
    """1300 boxes whose symmetric work units together pass 2^31: the batch itself is within every limit."""
    assert _lib.nf_workspace_bytes_batched(batch(1300, 10 ** 6, 25, 4)) > 0


@pytest.mark.parametrize("R", [1, 2, 3, 4])
@pytest.mark.parametrize("N,K", [(1 << 20, 25), (1 << 25, 80), (1 << 27, 128), (1 << 28, 160)])
def test_one_box(N, K, R):
    need = _lib.nf_workspace_bytes(N, K, R)
    # the planes of a box are within 80 GB and may take the place of its rows
    assert 0 < need <= 1.05 * directed_bytes(N, K, R) + 84e9, need


def test_sorting_alone_needs_no_partial_sums():
    # keys 8, offsets between passes 16, offsets 16, permutation 4, and the sort's counts (one word per digit value
    # and tile of 2048 particles, 9-bit digits at most): 45 bytes a particle; the cells' offsets
    for N, K in ((60000000, 100), (20000000, 64), (1000, 4)):
        need = _lib.nf_bin_workspace_bytes(N, K)
        assert 0 < need <= 45.5 * N + 4 * K ** 3 + 65536, (N, K, need)
    assert _lib.nf_bin_workspace_bytes(0, 8) == 0 and _lib.nf_bin_workspace_bytes(1000, 1291) == 0


@pytest.mark.gpu
def test_binning_keeps_a_workspace_of_its_own_size():
    import torch
    import paper_2110_11392_gb300 as nf
    from paper_2110_11392_gb300 import nearfield
    nearfield._WS_CACHE.clear()
    N, K = 1 << 20, 25
    pos = torch.rand((N, 3), device="cuda")
    nf.bin_particles(pos, 1.0, K)
    nf.multipoles(pos, 1.0, K, 2)
    assert nf.workspace(0).numel() == _lib.nf_bin_workspace_bytes(N, K)
    nf.forces(pos, 1.0, K, 2, 1e-4)  # grows it
    assert nf.workspace(0).numel() == _lib.nf_workspace_bytes(N, K, 2)

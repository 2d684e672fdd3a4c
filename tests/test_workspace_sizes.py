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
    # 5 % for the tables per cell, the sort's counts and the work units of one round
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

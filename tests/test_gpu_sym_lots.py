"""A batch whose symmetric boxes do not fit side by side in the shared partial sums runs in lots: bit for bit the
single calls, forward (with the net force), adjoint and replayed from a graph."""
import numpy as np
import pytest

from workloads import uniform_positions, upstream_gradient

from _helpers import to_dev

pytestmark = pytest.mark.gpu


def test_lots_equal_single_calls():
    import torch
    import paper_2110_11392_gb300 as nf
    from paper_2110_11392_gb300 import _lib
    # 2.5 GB of planes each for the large boxes (113 slots): three fit in 8 GiB, so there are two lots, with
    # directed boxes in both
    parts = [(1400003, 30, 4), (5000, 9, 2), (1400001, 30, 4), (1399999, 30, 4), (1400007, 30, 4), (4001, 9, 4)]
    pos = [uniform_positions(N, q + 1) for q, (N, _, _) in enumerate(parts)]
    boxes = [dict(N=N, K=K, R=R, eps=2e-4, box=1.0) for N, K, R in parts]
    assert _lib.nf_workspace_bytes_batched(boxes) < 4 * _lib.nf_workspace_bytes(1399999, 30, 4)
    cat = to_dev(np.concatenate(pos))
    run = nf.BatchedNearField(boxes, net=True)
    acc, net = run(cat).clone(), run.net.clone()
    g = to_dev(upstream_gradient(len(cat), 8))
    grad = torch.empty_like(cat)
    _lib.nf_forces_adjoint_batched(run.arr, cat, g, grad, None, run.ws)
    directed = torch.empty_like(cat)
    _lib.nf_forces_batched(run.arr, cat, directed, None, (4, 128, 4, 0), run.ws)
    off = 0
    for q, (N, K, R) in enumerate(parts):
        s = slice(off, off + N)
        x, gx = cat[s].contiguous(), g[s].contiguous()
        one, n1 = nf.forces(x, 1.0, K, R, 2e-4, net=True)
        assert torch.equal(acc[s], one) and torch.equal(net[q], n1), q
        assert torch.equal(grad[s], nf.forces_adjoint(x, gx, 1.0, K, R, 2e-4)), q
        assert torch.equal(directed[s], one) == (N < 10000), q
        off += N
    run.capture()
    acc.zero_()
    assert torch.equal(run(cat), directed) is False
    for q, (N, K, R) in enumerate(parts):
        s = slice(sum(p[0] for p in parts[:q]), sum(p[0] for p in parts[:q + 1]))
        assert torch.equal(run.acc[s], nf.forces(cat[s].contiguous(), 1.0, K, R, 2e-4)), q

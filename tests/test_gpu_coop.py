"""Cooperative items (the warps of a block share an item of the directed kernel): bit-identical to one warp
per item, which a batch with enough boxes runs, at every size class of the rule, ragged numbers of stages,
empty cells and every radius; forward with net force, adjoint, density, and the time step."""
import numpy as np
import pytest

import oracle
from workloads import clustered_positions, uniform_positions, upstream_gradient
from workloads.recipes import Workload, plummer_eps

from _helpers import assert_force_parity, sample_sinks, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K,R", [(1, 5, 2), (300, 5, 2), (4097, 5, 2), (7000, 7, 3), (12000, 9, 4), (16384, 6, 1),
                                   (30001, 8, 3), (40000, 12, 2), (65536, 10, 2), (131073, 13, 2)])
def test_equal_to_one_warp_per_item(N, K, R):
    import torch
    import paper_2110_11392_gb300 as nf
    from paper_2110_11392_gb300 import _lib
    x = clustered_positions(N, K, N) if N % 2 else uniform_positions(N, N)
    eps = plummer_eps(N) if N > 100 else 1e-3
    pos, g = to_dev(x), to_dev(upstream_gradient(N, 2))
    acc, net = nf.forces(pos, 1.0, K, R, eps, net=True)
    grad = nf.forces_adjoint(pos, g, 1.0, K, R, eps)
    # the same box beside one of 2 * 10^5 particles that fills the chip with items
    other = uniform_positions(200000, 5)
    boxes = [dict(N=N, K=K, R=R, eps=eps, box=1.0), dict(N=len(other), K=15, R=2, eps=1e-3, box=1.0)]
    cat = torch.cat([pos, to_dev(other)])
    run = nf.BatchedNearField(boxes, net=True)
    both = run(cat)
    assert torch.equal(both[:N], acc) and torch.equal(run.net[0], net)
    gb = torch.empty_like(cat)
    _lib.nf_forces_adjoint_batched(run.arr, cat, torch.cat([g, to_dev(other)]), gb, None, run.ws)
    assert torch.equal(gb[:N], grad)
    # density: the same accelerations, and both modes agree
    rhos = []
    try:
        for mode in (_lib.NF_DENS_FUSED, _lib.NF_DENS_DEFERRED):
            _lib.nf_set_density_mode(mode)
            a, rho = nf.forces_density(pos, 1.0, K, R, eps, 0.2 / K)
            assert torch.equal(a, acc)
            rhos.append(rho)
    finally:
        _lib.nf_set_density_mode(_lib.NF_DENS_AUTO)
    assert torch.equal(*rhos)
    w = Workload("coop", x, 1.0, K, R, eps)
    idx = sample_sinks(w, 1000, seed=N, include_densest=False)
    if N > 1:
        assert_force_parity(acc.cpu().numpy()[idx], oracle.forces(x, 1.0, K, R, eps, sinks=idx), label=f"{N} {K} {R}")
    ref = oracle.density(x, 1.0, K, R, 0.2 / K, sinks=idx)
    assert (np.abs(rhos[0].cpu().numpy()[idx] - ref) <= 1e-4 * ref).all()


def test_capture_and_explicit_shape():
    """The choice is part of a captured graph, and an explicit tuning of the same sums gives the same bits."""
    import torch
    import paper_2110_11392_gb300 as nf
    x = uniform_positions(5000, 3)
    box = [dict(N=5000, K=5, R=2, eps=1e-3, box=1.0)]
    pos = to_dev(x)
    acc = nf.forces(pos, 1.0, 5, 2, 1e-3)
    assert torch.equal(nf.BatchedNearField(box, tune=(4, 128, 4, 0))(pos), acc)
    graph = nf.BatchedNearField(box).capture()
    assert torch.equal(graph(pos), acc)

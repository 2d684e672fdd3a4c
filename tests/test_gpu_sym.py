"""The symmetric pair kernel (boxes of 2^18 particles and more under the built-in tuning) against the
FP64 oracle on sampled particles and against the directed kernel (an explicit tuning) on all of them:
ragged N, every radius, odd grids and boxes, empty regions, pencils that are cut into one-sided units,
close pairs across faces, a softening wider than a cell, batches of both kinds of box.  Boxes with much
of their work in a few pencils, that fill its lanes badly, or are small enough for nf_forces_noalloc's
scratch, run directed, bit for
bit as an explicit tuning of the same shape."""
import numpy as np
import pytest

import oracle
from workloads import clustered_positions, uniform_positions, upstream_gradient
from workloads.recipes import Workload

from _helpers import FORCE_MAX, FORCE_MEDIAN, assert_force_parity, dense_pencil_with_close_pairs, sample_sinks, to_dev

pytestmark = pytest.mark.gpu

N0 = 1 << 18
DIRECTED = (4, 128, 4, 0)  # the built-in shape's sums (four sinks per lane, stages of 128), directed


def one_cell(N, seed):
    rng = np.random.default_rng(seed)
    x = 0.5 + 0.01 * rng.standard_normal((N, 3))
    return (x % 1.0).astype(np.float32)


def blobs(N, seed):
    """Two dense cells in an otherwise sparse box: their pencils are cut into one-sided units."""
    rng = np.random.default_rng(seed)
    x = rng.random((N, 3))
    x[: N // 3] = 0.31 + 0.012 * rng.standard_normal((N // 3, 3))
    x[N // 3: N // 2] = 0.36 + 0.012 * rng.standard_normal((N // 2 - N // 3, 3))
    return (x % 1.0).astype(np.float32)


def some_blobs(N, seed, part):
    """Uniform, with `part` of the particles in eight dense spots: some dear pencils in a box that
    stays on the symmetric kernel."""
    rng = np.random.default_rng(seed)
    x = rng.random((N, 3))
    n = int(part * N)
    x[:n] = rng.random((8, 3))[rng.integers(0, 8, n)] + 0.008 * rng.standard_normal((n, 3))
    return (x % 1.0).astype(np.float32)


def soft_faces(N, K, seed):
    """Uniform, with 3000 close pairs that straddle cell faces in x, y or z."""
    rng = np.random.default_rng(seed)
    x = rng.random((N, 3))
    for q in range(3000):
        a = rng.random(3)
        a[q % 3] = rng.integers(0, K) / K
        h = 3e-4 * np.eye(3)[q % 3]
        x[2 * q], x[2 * q + 1] = a - h, a + h + 1e-4 * rng.random(3)
    return (x % 1.0).astype(np.float32)


# name: (workload, kernel that the forward and the adjoint call run)
CASES = {
    "ragged_K5": (lambda: Workload("", uniform_positions(N0 + 77, 1), 1.0, 5, 2, 1e-4), "dir", "dir"),
    "R1": (lambda: Workload("", clustered_positions(N0, 13, 2), 1.0, 13, 1, 4e-4), "dir", "dir"),
    "R1_large": (lambda: Workload("", clustered_positions(320001, 9, 2), 1.0, 9, 1, 4e-4), "dir", "sym"),
    "R1_huge": (lambda: Workload("", uniform_positions(1500007, 4), 1.0, 16, 1, 2e-4), "sym", "sym"),
    "R3_box": (lambda: Workload("", uniform_positions(N0 + 1, 3, 3.7), 3.7, 11, 3, 1e-3), "sym", "sym"),
    "R4": (lambda: Workload("", clustered_positions(N0 + 33, 17, 4), 1.0, 17, 4, 4e-4), "sym", "sym"),
    "half_empty": (lambda: Workload("", uniform_positions(500001, 5) * np.float32(0.5), 1.0, 20, 2, 4e-4), "sym", "sym"),
    "one_cell": (lambda: Workload("", one_cell(N0, 6), 1.0, 5, 2, 1e-4), "dir", "dir"),
    "blobs": (lambda: Workload("", blobs(N0 + 5, 7), 1.0, 19, 2, 2e-4), "dir", "dir"),
    "dense_pencil": (lambda: Workload("", dense_pencil_with_close_pairs(8, 6, 44000, 200), 1.0, 6, 2, 0.002),
                     "dir", "dir"),
    "wide_softening": (lambda: Workload("", uniform_positions(N0 + 9, 9), 1.0, 11, 2, 1.5 / 11 / 2.16), "sym", "sym"),
    "some_blobs": (lambda: Workload("", some_blobs(N0 + 21, 10, 0.1), 1.0, 11, 2, 3e-4), "sym", "sym"),
    "few_blobs": (lambda: Workload("", some_blobs(N0 + 2, 11, 0.06), 1.0, 12, 2, 3e-4), "sym", "sym"),
    "soft_faces": (lambda: Workload("", soft_faces(N0 + 15, 11, 12), 1.0, 11, 2, 0.002), "sym", "sym"),
}


def directed(w, g=None):
    import torch
    from paper_2110_11392_gb300 import _lib
    box = dict(N=w.N, K=w.K, R=w.R, eps=w.eps, box=w.box)
    ws = torch.empty(_lib.nf_workspace_bytes_batched([box]), dtype=torch.uint8, device="cuda")
    pos = to_dev(w.pos)
    out = torch.empty_like(pos)
    if g is None:
        _lib.nf_forces_batched(_lib.make_boxes([box]), pos, out, None, DIRECTED, ws)
    else:
        _lib.nf_forces_adjoint_batched(_lib.make_boxes([box]), pos, to_dev(g), out, DIRECTED, ws)
    return out.cpu().numpy().astype(np.float64)


@pytest.mark.parametrize("name", list(CASES))
def test_forces_and_net(name):
    import torch
    import paper_2110_11392_gb300 as nf
    make, kernel, _ = CASES[name]
    w = make()
    acc, net = nf.forces(to_dev(w.pos), w.box, w.K, w.R, w.eps, net=True)
    a = acc.cpu().numpy()
    d = directed(w)
    assert np.array_equal(a, d) == (kernel != "sym")
    if kernel != "sym":
        return
    idx = sample_sinks(w, 200, seed=1, include_densest=False)
    assert_force_parity(a[idx], oracle.forces(w.pos, w.box, w.K, w.R, w.eps, sinks=idx), label=name)
    # against the directed kernel on every particle: medians within twice the bar of each other, and
    # where the two differ most the oracle decides (the symmetric kernel keeps the bar there; the
    # directed one, with longer chains of sums, can pass it on forces that nearly cancel)
    err = np.linalg.norm(a - d, axis=1) / np.maximum(np.linalg.norm(d, axis=1), 1e-30)
    assert np.median(err) <= 2 * FORCE_MEDIAN, (name, np.median(err))
    worst = np.sort(np.argsort(-err)[:300])
    exact = oracle.frac_error(a[worst], oracle.forces(w.pos, w.box, w.K, w.R, w.eps, sinks=worst))
    assert exact.max() <= FORCE_MAX, (name, exact.max())
    bound = w.N * 2.0 ** -52 * np.abs(a.astype(np.float64)).sum(0) / w.N
    assert (np.abs(net.cpu().numpy() - a.astype(np.float64).sum(0) / w.N) <= bound).all()
    again = nf.forces(to_dev(w.pos), w.box, w.K, w.R, w.eps)
    assert torch.equal(again, acc)
    from paper_2110_11392_gb300 import _lib
    assert _lib.nf_status_read(nf.workspace(0)) == _lib.NF_OK


@pytest.mark.parametrize("name", list(CASES))
def test_adjoint(name):
    import paper_2110_11392_gb300 as nf
    make, _, kernel = CASES[name]
    w = make()
    g = upstream_gradient(w.N, 3)
    grad = nf.forces_adjoint(to_dev(w.pos), to_dev(g), w.box, w.K, w.R, w.eps).cpu().numpy()
    d = directed(w, g)
    assert np.array_equal(grad, d) == (kernel != "sym")
    if kernel != "sym":
        return
    idx = sample_sinks(w, 100, seed=2, include_densest=False)
    ref = oracle.adjoint(w.pos, g.astype(np.float64), w.box, w.K, w.R, w.eps, sinks=idx)
    # the bar of the directed adjoint (median 1e-5 of the gradient), and twice that between the kernels
    assert np.median(oracle.frac_error(grad[idx], ref)) <= 1e-5
    size = np.linalg.norm(d, axis=1)
    err = np.linalg.norm(grad - d, axis=1) / np.maximum(size, 1e-3 * np.median(size))
    assert np.median(err) <= 2e-5, (name, np.median(err))


@pytest.mark.parametrize("name,b_cells", [("R1_huge", 0.2), ("R3_box", 0.6), ("some_blobs", 0.05), ("half_empty", 1.7)])
def test_density_modes_and_same_forces(name, b_cells):
    import torch
    import paper_2110_11392_gb300 as nf
    from paper_2110_11392_gb300 import _lib
    w = CASES[name][0]()
    pos, b = to_dev(w.pos), b_cells * w.box / w.K
    b = min(b, w.R * w.box / w.K)
    acc = nf.forces(pos, w.box, w.K, w.R, w.eps)
    rhos = []
    try:
        for mode in (_lib.NF_DENS_FUSED, _lib.NF_DENS_DEFERRED):
            _lib.nf_set_density_mode(mode)
            a, rho = nf.forces_density(pos, w.box, w.K, w.R, w.eps, b)
            assert torch.equal(a, acc)
            rhos.append(rho)
    finally:
        _lib.nf_set_density_mode(_lib.NF_DENS_AUTO)
    assert torch.equal(*rhos)
    idx = sample_sinks(w, 200, seed=3, include_densest=False)
    ref = oracle.density(w.pos, w.box, w.K, w.R, b, sinks=idx)
    err = np.abs(rhos[0].cpu().numpy()[idx] - ref) / ref
    assert np.median(err) <= 1e-6 and err.max() <= 1e-4


def test_batch_of_both_kinds_equals_single_calls():
    import torch
    import paper_2110_11392_gb300 as nf
    from paper_2110_11392_gb300 import _lib
    parts = [(uniform_positions(5000, 1), 5, 2), (clustered_positions(N0 + 3, 16, 2), 16, 2),
             (uniform_positions(N0 - 1, 3), 17, 1), (uniform_positions(N0, 4), 12, 3)]
    boxes = [dict(N=len(x), K=K, R=R, eps=4e-4, box=1.0) for x, K, R in parts]
    pos = to_dev(np.concatenate([x for x, _, _ in parts]))
    run = nf.BatchedNearField(boxes, net=True)
    acc, net = run(pos).clone(), run.net.clone()
    g = to_dev(upstream_gradient(len(pos), 8))
    grad = torch.empty_like(pos)
    _lib.nf_forces_adjoint_batched(run.arr, pos, g, grad, None, run.ws)
    off = 0
    for q, (x, K, R) in enumerate(parts):
        s = slice(off, off + len(x))
        one, n1 = nf.forces(pos[s].contiguous(), 1.0, K, R, 4e-4, net=True)
        assert torch.equal(acc[s], one) and torch.equal(net[q], n1)
        assert torch.equal(grad[s], nf.forces_adjoint(pos[s].contiguous(), g[s].contiguous(), 1.0, K, R, 4e-4))
        off += len(x)
    run.capture()
    assert torch.equal(run(pos), acc)


def test_guards_stay_intact():
    import torch
    import paper_2110_11392_gb300 as nf  # noqa: F401
    from paper_2110_11392_gb300 import _lib
    w = CASES["some_blobs"][0]()
    _lib.nf_set_debug(True)
    try:
        ws = torch.empty(_lib.nf_workspace_bytes(w.N, w.K, w.R), dtype=torch.uint8, device="cuda")
        pos = to_dev(w.pos)
        out, rho = torch.empty_like(pos), torch.empty(w.N, device="cuda")
        _lib.nf_forces(pos, w.box, w.K, w.R, w.eps, out, None, ws)
        assert _lib.nf_status_read(ws) == _lib.NF_OK
        _lib.nf_forces_adjoint(pos, pos, w.box, w.K, w.R, w.eps, out, ws)
        assert _lib.nf_status_read(ws) == _lib.NF_OK
        _lib.nf_forces_density(pos, w.box, w.K, w.R, w.eps, 0.01, out, rho, ws)
        assert _lib.nf_status_read(ws) == _lib.NF_OK
    finally:
        _lib.nf_set_debug(False)

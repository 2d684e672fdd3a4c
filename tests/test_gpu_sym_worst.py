"""The symmetric pair kernel on its hardest particles: every particle of the densest cell, and the 300 particles
whose symmetric and directed results differ most, against the FP64 oracle; forward, adjoint and density.  The
boxes hold dear pencils that are cut into one-sided units, wide stencils, empty regions and close pairs."""
import numpy as np
import pytest

import oracle
from workloads import upstream_gradient

from _helpers import FORCE_MAX, FORCE_MEDIAN, assert_force_parity, sample_sinks, to_dev
from test_gpu_adjoint import ADJ_MAX, ADJ_MEDIAN
from test_gpu_sym import CASES, directed

pytestmark = pytest.mark.gpu


def worst(a, d, count=300):
    """The particles whose results differ most, by the size of the difference."""
    return np.sort(np.argsort(-np.linalg.norm(a.astype(np.float64) - d, axis=1))[:count])


@pytest.mark.parametrize("name", [n for n, c in CASES.items() if c[1] == "sym"])
def test_forces(name):
    import paper_2110_11392_gb300 as nf
    w = CASES[name][0]()
    a = nf.forces(to_dev(w.pos), w.box, w.K, w.R, w.eps).cpu().numpy()
    idx = np.union1d(sample_sinks(w, 100, seed=4), worst(a, directed(w)))
    assert_force_parity(a[idx], oracle.forces(w.pos, w.box, w.K, w.R, w.eps, sinks=idx), label=name)


@pytest.mark.parametrize("name", [n for n, c in CASES.items() if c[2] == "sym"])
def test_adjoint(name):
    import paper_2110_11392_gb300 as nf
    w = CASES[name][0]()
    g = upstream_gradient(w.N, 5)
    a = nf.forces_adjoint(to_dev(w.pos), to_dev(g), w.box, w.K, w.R, w.eps).cpu().numpy()
    idx = np.union1d(sample_sinks(w, 100, seed=5), worst(a, directed(w, g)))
    ref = oracle.adjoint(w.pos, g.astype(np.float64), w.box, w.K, w.R, w.eps, sinks=idx)
    size = np.linalg.norm(ref, axis=1)
    err = np.linalg.norm(a[idx] - ref, axis=1) / np.maximum(size, 1e-2 * np.median(size))
    assert np.median(err) <= ADJ_MEDIAN and err.max() <= ADJ_MAX, (name, np.median(err), err.max())


@pytest.mark.parametrize("name,b_cells", [("R1_huge", 0.5), ("R3_box", 0.6), ("some_blobs", 0.3), ("half_empty", 1.7)])
def test_density(name, b_cells):
    import paper_2110_11392_gb300 as nf
    w = CASES[name][0]()
    b = b_cells * w.box / w.K
    _, rho = nf.forces_density(to_dev(w.pos), w.box, w.K, w.R, w.eps, b)
    idx = sample_sinks(w, 200, seed=6)
    ref = oracle.density(w.pos, w.box, w.K, w.R, b, sinks=idx)
    err = np.abs(rho.cpu().numpy()[idx] - ref) / ref
    assert np.median(err) <= FORCE_MEDIAN and err.max() <= FORCE_MAX, (name, np.median(err), err.max())

"""The symmetric pair kernel is no further from 64 bits than the directed one: mean fractional error over the same
40,000 particles, uniform boxes (in which one chain of sums over all tiles of a pencil was 3 to 8 % further off)."""
import numpy as np
import pytest

import oracle
from workloads import uniform_positions, upstream_gradient
from workloads.recipes import Workload

from _helpers import to_dev
from test_gpu_sym import directed

pytestmark = pytest.mark.gpu

# a mean of 40,000 errors whose spread is about their size is known to 0.5 %, a ratio of two to 0.7 %: 2 % are three of these
MARGIN = 1.02


@pytest.mark.parametrize("adjoint,N,K,R", [(False, 36000001, 83, 2), (False, 2097155, 32, 2), (True, 2097155, 32, 3),
                                           (True, 1400003, 28, 2)])
def test_mean_error(adjoint, N, K, R):
    import paper_2110_11392_gb300 as nf
    w = Workload("", uniform_positions(N, 11), 1.0, K, R, 1.0 / (40 * N ** (1 / 3)))
    idx = np.sort(np.random.default_rng(2).choice(N, 40000, replace=False))
    if adjoint:
        g = upstream_gradient(N, 3)
        a, d = nf.forces_adjoint(to_dev(w.pos), to_dev(g), 1.0, K, R, w.eps).cpu().numpy(), directed(w, g)
        ref = oracle.adjoint(w.pos, g.astype(np.float64), 1.0, K, R, w.eps, sinks=idx)
    else:
        a, d = nf.forces(to_dev(w.pos), 1.0, K, R, w.eps).cpu().numpy(), directed(w)
        ref = oracle.forces(w.pos, 1.0, K, R, w.eps, sinks=idx)
    assert not np.array_equal(a, d)
    sym, one = oracle.frac_error(a[idx], ref).mean(), oracle.frac_error(d[idx], ref).mean()
    assert sym <= MARGIN * one, (sym, one)

"""The packed double-float kernels of the far field where pairs of particles break: odd counts, one
particle, cells of one and of chunk-edge occupancies, every order.  Double-float against the FP64 mode,
to the 1e-12 of the largest value that the two arithmetics keep."""
import numpy as np
import pytest

from workloads import uniform_positions

from _helpers import to_dev

pytestmark = pytest.mark.gpu


def occupancies(K, seed):
    """Cells of 0, 1, 2, 3, 31, 32, 33, 63, 64, 65 and 129 particles."""
    rng = np.random.default_rng(seed)
    want = [0, 1, 2, 3, 31, 32, 33, 63, 64, 65, 129]
    parts = []
    for q, n in enumerate(want):
        c = np.array([q % K, (q // K) % K, (3 * q) % K])
        parts.append((c + rng.random((n, 3))) / K)
    return np.concatenate(parts).astype(np.float32)


@pytest.mark.parametrize("p", [0, 1, 2, 3, 5, 8, 11, 12])
@pytest.mark.parametrize("kind", ["one", "odd", "cells"])
def test_double_float_equals_fp64(p, kind):
    import torch
    import paper_2110_11392_gb300 as nf
    from paper_2110_11392_gb300 import _lib
    K = 8 if p % 2 else 7
    x = {"one": lambda: uniform_positions(1, 3), "odd": lambda: uniform_positions(2049, 4),
         "cells": lambda: occupancies(K, p)}[kind]()
    f = nf.FarField(K, 2, p)
    pos = to_dev(x)
    df, tdf = f(pos, want_taylors=True)
    try:
        _lib.nf_far_set_arith(_lib.NF_FAR_FP64)
        ref, tref = f(pos, want_taylors=True)
    finally:
        _lib.nf_far_set_arith(_lib.NF_FAR_DOUBLE_FLOAT)
    torch.cuda.synchronize()
    top = max(float(ref.abs().max()), float(tref.abs().max()) / max(1, len(x)))
    assert float((df - ref).abs().max()) <= 1e-12 * top
    # adding into FP32 rounds the same values once
    add = torch.zeros(len(x), 3, device="cuda")
    f(pos, add_to=add, want_far=False)
    assert torch.equal(add, df.float())

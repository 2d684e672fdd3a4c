"""The mixed-radix transforms where a thread takes one output of a large prime radix and a block takes lines
of several planes: prime lengths, a large prime after smaller factors (twiddles of a later step), one and many
lines to a block with a ragged last one, and the rebuild's level starts at the lowest orders."""
import numpy as np
import pytest

import oracle

from _helpers import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("arith", [0, 1], ids=["fp64", "double-float"])
@pytest.mark.parametrize("K,R,p", [(5, 2, 1), (7, 2, 2), (11, 1, 3), (14, 1, 4), (17, 2, 3), (22, 2, 3), (26, 2, 2),
                                   (33, 2, 2)])
def test_taylors_match_oracle(K, R, p, arith):
    import torch
    import paper_2110_11392_gb300 as nf
    from paper_2110_11392_gb300 import _lib
    pos = np.random.default_rng(K).random((3000, 3)).astype(np.float32)
    pos[pos >= 1.0] = 0.0
    before = _lib.nf_far_get_arith()
    _lib.nf_far_set_arith(arith)
    try:
        a, T = nf.FarField(K, R, p)(to_dev(pos), want_taylors=True)
        torch.cuda.synchronize()
    finally:
        _lib.nf_far_set_arith(before)
    aref, Tref = oracle.far_field(pos, 1.0, K, R, p, return_taylors=True)
    T = T.cpu().numpy()
    assert (np.abs(T - Tref).max(axis=0) / (np.abs(Tref).max(axis=0) + 1e-300)).max() < 1e-10
    assert np.abs(a.cpu().numpy() - aref).max() < 1e-10 * np.abs(aref).max()

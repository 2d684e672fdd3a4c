"""The binning's short cell rule (float pairs, nf_cell.cuh) on the CPU against the FP64 rule t = x K/box,
c = floor(t), offset = fp32((t - c) - 1/2): wherever the counting form or the sorting form accepts a value, its
cell and offset are the rule's, so the two can never disagree.  Values at and next to cell faces, inside and
outside the box."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2110_11392_gb300", "csrc")

# grids with faces where K/box times the coordinate, in FP32, lies on the other side of the face
FACES = [(32, 3.7), (64, 3.7), (128, 3.7), (31, 3.7), (34, 250.0), (68, 500.0), (109, 205.0), (101, 0.7), (183, 0.7),
         (155, 0.3), (199, 0.3), (177, 1.3), (212, 13.0), (8, 330.0), (127, 879.0), (75, 231.6), (101, 500.0)]


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    lib = str(tmp_path_factory.mktemp("cell") / "cell_rule.so")
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-fPIC", "-shared", "-I", CSRC,
                           os.path.join(HERE, "cell_rule_host.cpp"), "-o", lib])
    fn = ctypes.CDLL(lib).cell_rule

    def run(x, kl):
        n = len(x)
        out = [np.zeros(n, t) for t in (np.uint8, np.int32, np.uint8, np.int32, np.float32)]
        fn(x.ctypes.data_as(ctypes.c_void_p), ctypes.c_int64(n), ctypes.c_double(kl),
           *[o.ctypes.data_as(ctypes.c_void_p) for o in out])
        return out
    return run


def beside(v, ulps):
    """The FP32 values within `ulps` units in the last place of v > 0."""
    b = np.asarray(v, np.float64).astype(np.float32).view(np.int32)
    return (b[:, None] + np.arange(-ulps, ulps + 1, dtype=np.int32)).view(np.float32).ravel()


def check(rule, x, K, box):
    kl = K / box
    x = np.ascontiguousarray(x[x > 0])
    t = x.astype(np.float64) * kl
    c = np.floor(t)
    off = ((t - c) - 0.5).astype(np.float32)
    ok1, c1, ok2, c2, o2 = rule(x, kl)
    ok1, ok2 = ok1 != 0, ok2 != 0
    assert np.array_equal(c1[ok1], c[ok1]), (K, box, x[ok1][c1[ok1] != c[ok1]][:3])
    assert np.array_equal(c2[ok2], c[ok2]), (K, box, x[ok2][c2[ok2] != c[ok2]][:3])
    assert np.array_equal(o2[ok2].view(np.int32), off[ok2].view(np.int32)), (K, box)
    return ok1, ok2


@pytest.mark.parametrize("K,box", FACES)
def test_every_face(rule, K, box):
    w = box / K
    k = np.concatenate([np.arange(1, 8 * K + 1), np.unique(np.logspace(3, 6, 3000).astype(int))])
    check(rule, beside(k * w, 6), K, box)
    check(rule, beside((k - 0.5) * w, 6), K, box)


def test_faces_of_random_grids(rule):
    rng = np.random.default_rng(5)
    for q in range(4000):
        K = int(rng.integers(1, 256))
        box = float(round(10.0 ** rng.uniform(-1, 3), int(rng.integers(0, 4))) or 0.5)
        check(rule, beside(np.arange(1, 2 * K + 1) * (box / K), 6), K, box)


@pytest.mark.parametrize("K,box", FACES)
def test_plain_values_take_the_short_rule(rule, K, box):
    """The rule is not only right but used: of a uniform box's coordinates it leaves out 2 x 2^-22 p (p up to K)
    at the faces and those below 2^-12 of a cell, less than 1e-3 in all."""
    x = (np.random.default_rng(1).random(200000) * box).astype(np.float32)
    ok1, _ = check(rule, x, K, box)
    assert ok1.mean() > 0.999

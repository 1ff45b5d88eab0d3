"""Sine and cosine of a uniform draw's angle by the table against quadruple precision: the tabulated value and the last sum
round once each, the series' tails and the small terms leave less than one rounding more, so 2^-51; and beside the axes,
where the table's entries are exact zeros, 2^-50 of the value itself.  Draws at every tabulated angle and half way between
them, at both ends of the range, and random ones."""
import ctypes as C

import numpy as np
import pytest

from paper_1504_06570_gb300 import phosim as P

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


def evaluate(op, a):
    out, dp = np.zeros(len(a)), C.POINTER(C.c_double)
    assert P.lib().phosim_fp64_eval(op, a.ctypes.data_as(dp), out.ctypes.data_as(dp), len(a)) == 0
    return out


def test_sincos_of_a_draw():
    if np.finfo(np.longdouble).nmant < 100:
        pytest.skip("no quadruple precision on this machine")
    rng = np.random.default_rng(12)
    steps = np.arange(512, dtype=np.uint64) * np.uint64(2 ** 23)
    w = np.unique(np.r_[rng.integers(0, 2 ** 32, 100000, dtype=np.uint64), steps, (steps + np.uint64(2 ** 32 - 1)) % np.uint64(2 ** 32),
                        steps + np.uint64(1), np.uint64(2 ** 32 - 1)])
    a = w.astype(np.float64)
    turn = (2 * w.astype(np.longdouble) + 1) / np.longdouble(2) ** 33
    pi = np.longdouble("3.14159265358979323846264338327950288")
    eighth = np.rint(8 * turn)                    # reduced exactly: the reference keeps its relative accuracy at the axes
    x = 2 * pi * (turn - eighth / 8)
    s, c, h, q = np.sin(x), np.cos(x), np.sqrt(np.longdouble(0.5)), eighth.astype(int) % 8
    ks = np.array([0, h, 1, h, 0, -h, -1, -h], np.longdouble)[q]
    kc = np.array([1, h, 0, -h, -1, -h, 0, h], np.longdouble)[q]
    for op, exact in ((15, s * kc + c * ks), (16, c * kc - s * ks)):
        err = np.abs(evaluate(op, a) - exact)
        assert np.max(err) < 2.0 ** -51
        near = np.abs(exact) < 0.01
        assert near.sum() > 100 and np.max(err[near] / np.abs(exact[near])) < 2.0 ** -50

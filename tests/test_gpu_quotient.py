"""The single-precision quotient and root by one correction with the exact remainder, against the correctly rounded values:
the remainder of a quotient or root off by 2^-22 leaves 2^-44 of the value before the last rounding, so the result is the
correctly rounded one unless the value lies that close to the middle of two floats (2^-44 of a spacing of 2^-24: one in
1e6, and at most 1 in 1e4 asked for here), and then its neighbour."""
import ctypes as C

import numpy as np
import pytest

from paper_1504_06570_gb300 import phosim as P

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


def evaluate(op, a, k=1.0):
    a = np.ascontiguousarray(a, np.float64)
    out, dp = np.full(len(a), k), C.POINTER(C.c_double)
    assert P.lib().phosim_fp64_eval(op, a.ctypes.data_as(dp), out.ctypes.data_as(dp), len(a)) == 0
    return out


@pytest.mark.parametrize("k", [1.0, 3.0, -0.7, 1.9999999, 1e-12, -7e9, 1.25e-5])
def test_quotient_and_root(k):
    rng = np.random.default_rng(11)
    a = (10.0 ** rng.uniform(-12, 12, 100000) * rng.uniform(1, 10, 100000)).astype(np.float32).astype(np.float64)
    signed = np.r_[a * rng.choice([-1.0, 1.0], a.size), 0.0]
    for got, exact in ((evaluate(12, signed, k), signed / np.float64(np.float32(k))), (evaluate(13, a * abs(k)), None)):
        if exact is None:
            exact = np.sqrt((a * abs(k)).astype(np.float32).astype(np.float64))
        near = exact.astype(np.float32)
        assert np.mean(got == near) >= 1.0 - 1e-4
        assert np.all(np.abs(got - near) <= np.spacing(np.abs(near)))

"""The logarithm of a uniform draw by its table against extended precision: the table's entries, the product with the
table's reciprocal (exact), the series and three sums leave three roundings and a truncation below 2^-53, so 2^-51 of the
value (also just below 1, where the value is small), at every table entry's edges, at both ends and at random draws.  The
dense reference in double, log1p or log of the exact draw, may itself be off by 2^-52."""
import ctypes as C
from decimal import Decimal, getcontext

import numpy as np
import pytest

from paper_1504_06570_gb300 import phosim as P

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


@pytest.mark.parametrize("n", [1, 200000])
def test_log_of_a_draw(n):
    getcontext().prec = 40
    rng = np.random.default_rng(8)
    w = rng.integers(0, 2 ** 32, n, dtype=np.uint64)
    if n > 1:
        edges = np.array([((256 + i) << k) >> 8 for k in range(8, 32) for i in range(256)], np.uint64)
        w = np.unique(np.r_[w, edges, edges - 1, np.arange(5, dtype=np.uint64), 2 ** 32 - 1 - np.arange(300, dtype=np.uint64),
                            (rng.random(2000) * 2.0 ** rng.uniform(0, 32, 2000)).astype(np.uint64)])
    a, dp = w.astype(np.float64), C.POINTER(C.c_double)
    out = np.zeros(len(a))
    assert P.lib().phosim_fp64_eval(14, a.ctypes.data_as(dp), out.ctypes.data_as(dp), len(a)) == 0
    u = (a + 0.5) * 2.0 ** -32
    ref = np.where(u > 0.5, np.log1p(-(2.0 ** 32 - 0.5 - a) * 2.0 ** -32), np.log(u))
    assert np.max(np.abs(out / ref - 1.0)) < 2.0 ** -51 + 2.0 ** -52
    for k in range(0, len(w), max(1, len(w) // 300)):
        exact = (Decimal(2 * int(w[k]) + 1) / Decimal(2 ** 33)).ln()
        assert abs(Decimal(out[k]) / exact - 1) < Decimal(2) ** -51

"""A screen coordinate's node and fraction by integers against exact rational arithmetic: the coordinate is cut at 2^-40 mm
and the fraction at 2^-52 of a pixel, so node + fraction lies within 2^-40 k + 2^-52 of s k (k, a double, is exact in the
form); the single-precision fraction within half a unit of its last place, or 2^-32, of that.  Pixels from 4 um to 16 km,
coordinates on and beside nodes, of both signs, tiny and up to the range's end (4 km), and past it.  And a screen that lies
beyond the range (its drift) against the same screen near the origin: the same image."""
import ctypes as C
from fractions import Fraction
from math import floor

import numpy as np
import pytest

from paper_1504_06570_gb300 import phosim as P
from tests import gpu_helpers as G

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


def split(op, a, k):
    a = np.ascontiguousarray(a, np.float64)
    out, dp = np.full(len(a), k), C.POINTER(C.c_double)
    assert P.lib().phosim_fp64_eval(op, a.ctypes.data_as(dp), out.ctypes.data_as(dp), len(a)) == 0
    return out


@pytest.mark.parametrize("pixel", [0.004, 0.3, 1.0, 40.0, 100.0, 2560.0, 5120.0, 1.6e7])
def test_node_and_fraction(pixel):
    rng = np.random.default_rng(5)
    k = 1.0 / pixel
    edge = rng.integers(-int(4e6 * k) - 1, int(4e6 * k) + 2, 200) * pixel
    edge = edge[np.abs(edge) < 4.19e6]
    s = np.r_[rng.uniform(-4.19e6, 4.19e6, 1500), rng.normal(size=500) * 1e3, rng.normal(size=200) * 10.0 ** rng.uniform(-15, 0, 200),
              edge, np.nextafter(edge, np.inf), np.nextafter(edge, -np.inf), 0.0, 2.0 ** 22 - 1.0, -2.0 ** 22 + 1.0]
    node, frac, single = split(9, s, k), split(10, s, k), split(11, s, k)
    assert np.array_equal(node, np.floor(node)) and np.all((frac >= 0.0) & (frac < 1.0))
    K, bound = Fraction(k), Fraction(2) ** -40 * Fraction(k) + Fraction(2) ** -52
    for x, i, f in zip(s, node, frac):
        assert abs(Fraction(i) + Fraction(f) - Fraction(x) * K) <= bound, (x, i, f)
    assert np.all(np.abs(single - frac) <= np.maximum(np.spacing(frac.astype(np.float32)) / 2, 2.0 ** -32))
    for far in (2.0 ** 22, -2.0 ** 22, 1e9, np.inf, np.nan):
        assert np.all(split(10, [far], k) == -1.0)
    assert np.all(split(10, [1.0], 1e6) == -1.0)


@pytest.mark.parametrize("precision", [P.PLAIN_FP64, P.MIXED])
def test_screen_beyond_the_range(precision):
    sc = G.test_system_scene(n_photons=20000)
    sc.sources.t0 = np.full(len(sc.sources.t0), 2.0 ** 23)
    sc.sources.t_exp = np.zeros(len(sc.sources.t0))
    for layer in sc.layers:
        layer.scales, layer.vx, layer.vy = layer.scales[:1], 0.0, 0.0
    still = G.run_gpu(sc, precision, moments=False)["rec"]
    for layer in sc.layers:                       # 256 nodes of 40 mm; 1280 mm/s for 2^23 s are 2^20 times as far
        layer.vx, layer.vy = 1280.0, -1280.0
    drift = G.run_gpu(sc, precision, moments=False)["rec"]
    both = ((still["flags"] & 1) & (drift["flags"] & 1)) == 1
    assert np.mean(still["flags"] == drift["flags"]) > 0.999 and both.sum() > 1000
    # the drifted coordinate is rounded at 2^33 mm: 2^-20 mm of a 40 mm pixel, 2.4e-8 of the gradient's step between
    # nodes; the images shift by at most that of the whole deflection (below 1 mm on the detector)
    for c in ("x", "y"):
        assert np.max(np.abs(still[c][both] - drift[c][both])) < 1e-6

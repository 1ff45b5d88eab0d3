"""Floors beyond 32 bits in the FP64 and mixed paths.  The floor and its integer around the ends of the range: given within
[-2^31, 2^31), refused outside it, also where the low 32 bits alone would look right.  A screen whose drifted coordinate is
2^31 to 2^32 pixels and more from the origin, in both directions, with sizes that are no power of two: the same photons as
the screen at rest, which a drift by whole screens leaves unchanged, in the trace and in the adjoint's forward pass.  And a
table read 2^31 to 2^32 nodes past its end: its last value."""
import ctypes as C

import numpy as np
import pytest

from paper_1504_06570_gb300 import inputs as I
from paper_1504_06570_gb300 import phosim as P
from tests import gpu_helpers as G

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


def test_floors_around_32_bits():
    b = 2.0 ** 31
    x = np.array([b - 1.0, b - 0.5, b, b + 0.5, b + 7.0, 1.5 * b, 2 * b - 1.0, 2 * b, 2 * b + 5.0, 3 * b, 4 * b, 1e15])
    x = np.r_[x, -x, np.nextafter(-b, 0.0), np.nextafter(-b, -np.inf), 0.0, -0.25, 2.2e9, -2.2e9]
    inside = (np.floor(x) >= -b) & (np.floor(x) < b)
    dp = C.POINTER(C.c_double)
    for op in (6, 7):
        out = np.ones(len(x))
        assert P.lib().phosim_fp64_eval(op, x.ctypes.data_as(dp), out.ctypes.data_as(dp), len(x)) == 0
        assert np.array_equal(out, np.where(inside, np.floor(x), 0.5))


def screens(n, turns):
    """One layer scale of n x n nodes of 40 mm, drifted by turns * 2^20 whole screens along x and back along y."""
    sc = G.test_system_scene(n_photons=20000)
    rng = np.random.default_rng(8)
    sc.sources.t0 = np.full(len(sc.sources.t0), 2.0 ** 20)
    sc.sources.t_exp = np.zeros(len(sc.sources.t0))
    for layer in sc.layers:
        layer.scales = [I.ScreenScale(40.0, I.phase_screen(n, 0.04, 0.15, 20.0, rng))]
        layer.vx, layer.vy = turns * n * 40.0, -turns * n * 40.0
    return sc


# the drift in pixels: n turns 2^20.  Its coordinate in millimetres is below 2^38, so it is rounded by 2^-16 mm, 4e-7 of a
# pixel, and moves a photon by that part of the change of a deflection (below 1 mm on the detector) from one node to the
# next, which is at most twice the deflection, once a layer: 2e-6 mm, with a factor of five.
@pytest.mark.parametrize("precision", [P.PLAIN_FP64, P.MIXED])
@pytest.mark.parametrize("n, turns", [(255, 9), (255, 18), (1500, 2), (1500, -2), (1500, 4), (255, -9), (256, 9), (256, 17)])
def test_screen_many_pixels_away(precision, n, turns):
    assert n * abs(turns) * 2 ** 20 >= 2 ** 31
    still = G.run_gpu(screens(n, 0), precision, moments=False)["rec"]
    drift = G.run_gpu(screens(n, turns), precision, moments=False)["rec"]
    both = ((still["flags"] & 1) & (drift["flags"] & 1)) == 1
    assert np.mean(still["flags"] == drift["flags"]) > 0.999 and both.sum() > 1000
    for c in ("x", "y"):
        assert np.max(np.abs(still[c][both] - drift[c][both])) < 1e-5


def test_adjoint_of_a_screen_many_pixels_away():
    out = []
    for turns in (0, 2):
        s = P.Scene(screens(1500, turns), P.PLAIN_FP64)
        out.append(s.grad(np.array([[1.0, 0.5, 0.0, 0.0, 0.0]]), [(1, 0), (1, 1)]))
        s.close()
    (g0, m0), (g1, m1) = out
    # at most a photon in a thousand crosses a limit (above), and moves the mean by its distance, below 1 mm, of them
    assert abs(m0[0, 0] - m1[0, 0]) <= 1e-3 * m0[0, 0] and np.all(np.abs(m0[0, 1:3] - m1[0, 1:3]) < 1e-3)
    assert np.all(np.abs(g0 - g1) <= 1e-3 * np.abs(g0).max())


def test_table_read_far_past_its_end():
    recs = []
    for ell in ([0.001, 0.03], [0.03, 0.03]):
        sc = G.test_system_scene(n_photons=20000)
        d = sc.detector
        # wavelengths of 450 to 650 nm lie (50 to 250 nm) / 6e-8 nm = 0.8e9 to 4.2e9 nodes from the first
        d.ell, d.ell_lam0, d.ell_dlam = np.array(ell), 400.0, 6e-8
        recs.append(G.run_gpu(sc, P.PLAIN_FP64, moments=False)["rec"])
    assert (recs[0]["flags"] & 1).sum() > 1000
    assert np.array_equal(recs[0], recs[1])

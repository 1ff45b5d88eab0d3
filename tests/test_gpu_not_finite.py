"""Values that are no numbers, or beyond single precision, on the FP64 and mixed paths: a photon without a direction or a
place is lost where Newton's method does not settle (an aspheric surface, as the oracle has it) or at the aperture (a
conic), and never detected; the others of its scene are as they are without it."""
import numpy as np
import pytest

from paper_1504_06570_gb300 import inputs as I
from paper_1504_06570_gb300 import phosim as P
from tests import gpu_helpers as G

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]

VIGNETTED, MISSED, NEWTON, NOT_CONVERTED = 1, 2, 3, 7
BOTH = pytest.mark.parametrize("precision", [P.PLAIN_FP64, P.MIXED])


def scene():
    return G.test_system_scene(sources=G.mixed_sources([4000, 3000, 2000], seed=4))


def reasons(rec):
    """(reason, surface) of every photon; (0, .) of a detected one."""
    return np.where(rec["flags"] & 1, 0, rec["flags"] >> 8 & 0xff), rec["flags"] >> 16


@BOTH
@pytest.mark.parametrize("width", [np.nan, np.inf, 3.0])
@pytest.mark.parametrize("figure", [True, False])
def test_photons_without_a_direction(precision, width, figure):
    # the second and third source's offsets: no numbers, or most of them beyond 1 rad
    sc = scene()
    sc.sources.a = np.full(3, width)
    if not figure:
        sc.surfaces[0].zern = ()
    rec = G.run_gpu(sc, precision, moments=False)["rec"]
    plain = scene()
    if not figure:
        plain.surfaces[0].zern = ()
    points = G.run_gpu(plain, precision, moments=False)["rec"]
    assert np.array_equal(rec[:4000], points[:4000])
    why, surface = reasons(rec[4000:])
    assert not np.any(why == 0)
    at_first = (why == (NEWTON if figure else VIGNETTED)) & (surface == 0)
    assert np.mean(at_first) > (0.5 if width == 3.0 else 0.999)
    assert not np.any((why == MISSED) & (surface == 0)) or width == 3.0



@BOTH
@pytest.mark.parametrize("t0, t_exp", [(np.nan, 15.0), (np.inf, 15.0), (-np.inf, 0.0), (0.0, np.inf), (0.0, np.nan)])
def test_photons_without_a_time(oracle_mod, precision, t0, t_exp):
    # no place on the drifting screens, so no kick and no direction
    sc = scene()
    sc.sources.t0, sc.sources.t_exp = np.full(3, t0), np.full(3, t_exp)
    rec = G.run_gpu(sc, precision, moments=False)["rec"]
    assert np.array_equal(rec["flags"], G.oracle_trace(oracle_mod, sc)["flags"]) and not np.any(rec["flags"] & 1)


@BOTH
@pytest.mark.parametrize("v", [1280.0, -1280.0])
def test_screen_too_far_for_a_fraction(oracle_mod, precision, v):
    # 2^60 s at 1280 mm/s: the coordinate is -+1280 2^60 mm whatever the photon's place, a node of the 256 of 40 mm
    sc = scene()
    sc.sources.t0, sc.sources.t_exp = np.full(3, 2.0 ** 60), np.zeros(3)
    for layer in sc.layers:
        layer.vx, layer.vy = v, -v
    gpu, ora = G.run_gpu(sc, precision, moments=False), G.oracle_trace(oracle_mod, sc)
    assert np.sum(ora["flags"] & 1) > 1000
    G.compare_records(sc, gpu, ora, pos_tol_px=1e-4)


def test_table_without_a_place(oracle_mod):
    # an absorption table that starts nowhere: no length, no conversion
    sc = scene()
    sc.detector.ell_lam0 = np.nan
    rec = G.run_gpu(sc, P.PLAIN_FP64, moments=False)["rec"]
    ora = G.oracle_trace(oracle_mod, sc)
    assert np.all((rec["flags"] == ora["flags"]) | G.boundary_mask(ora))
    assert not np.any(rec["flags"] & 1) and np.sum(reasons(rec)[0] == NOT_CONVERTED) > 1000


@BOTH
def test_glass_without_an_index(oracle_mod, precision):
    # blue-shifted to 40 to 70 nm, where the Sellmeier formula of silica has negative squares: no index, no direction, and
    # the next surface's aperture drops the photon; the others are the oracle's
    sc = scene()
    sc.sources.redshift = np.full(3, -0.9)
    rec = G.run_gpu(sc, precision, moments=False)["rec"]
    ora = G.oracle_trace(oracle_mod, sc)
    l2 = (rec["lam"] * 1e-3) ** 2
    square = 1.0 + sum(b * l2 / (l2 - c) for b, c in zip(I.FUSED_SILICA_B, I.FUSED_SILICA_C))
    why, surface = reasons(rec)
    met = ~((surface == 0) | ((surface == 1) & (why == VIGNETTED)))          # went into the lens
    none = met & (square < -1e-9)
    assert none.sum() > 3000 and np.all(why[none] == VIGNETTED) and np.all(surface[none] == 2)
    real = square > 1e-9
    assert real.sum() > 1000 and np.all(((rec["flags"] == ora["flags"]) | G.boundary_mask(ora))[real])


def test_gradients_beyond_single_precision():
    # a band of phases of 1e300 on every screen: gradients that are infinite in single precision, or none; the photons that
    # the FP64 path loses for their directions the mixed path loses as well
    sc = G.test_system_scene(sources=G.mixed_sources([4000, 3000, 2000], seed=4), hf=True)
    for q in [q for layer in sc.layers for q in layer.scales]:
        q.phase = q.phase.copy()
        q.phase[10:14, 20:60] = 1e300
    full, mixed = (G.run_gpu(sc, p, moments=False)["rec"] for p in (P.PLAIN_FP64, P.MIXED))
    why, surface = reasons(full)
    nowhere = (why == NEWTON) & (surface == 0)
    assert nowhere.sum() > 1000 and np.array_equal(mixed["flags"][nowhere], full["flags"][nowhere])
    assert np.sum(full["flags"] & 1) > 1000


@BOTH
def test_no_kick_beyond_single_precision(oracle_mod, precision):
    # a reference wavelength of 1e-300 nm: (lambda / lambda_ref)^(-1/5) is nothing, and no photon is deflected
    sc = scene()
    sc.lambda_ref = 1e-300
    rec = G.run_gpu(sc, precision, moments=False)["rec"]
    ora = G.oracle_trace(oracle_mod, sc)
    assert np.all((rec["flags"] == ora["flags"]) | G.boundary_mask(ora)) and np.sum(rec["flags"] & 1) > 1000

"""The dynamic transmission test's first stage (an interval of the wavelength draw, when no records are asked for)
against the test with records, which decides every photon by its wavelength: the same images and the same counts,
and the same detected photons as without the test.  Coatings: one band with edges on and off the SED's bins, two bands
(the interval has a hole), a band that reaches the grid's ends, one that lets nothing pass, two coated surfaces whose
bands overlap or not, angles; redshifted sources, and the bundles' rays."""
import numpy as np
import pytest

from paper_1504_06570_gb300 import inputs as I
from paper_1504_06570_gb300 import phosim as P
from tests import gpu_helpers as G

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


def band(lo, hi, lam0=400.0, dlam=1.0, n=300, T=0.9, n_theta=1):
    lam = lam0 + dlam * (np.arange(n) + 0.5)
    t = np.where((lam > lo) & (lam < hi), T, 0.0)
    return I.Coating(lam0=lam0, dlam=dlam, theta0=0.0, dtheta=0.2, table=np.repeat(t[:, None], n_theta, 1).copy())


def two_bands():
    c = band(430.0, 640.0)
    c.table[80:140] = 0.0
    return c


COATINGS = {
    "band": [band(450.0, 650.0)],
    "off the bins": [band(450.3, 649.6, lam0=399.85, dlam=0.3, n=1003)],
    "fine grid": [band(455.0, 457.0, lam0=454.0, dlam=0.01, n=400)],
    "two bands": [two_bands()],
    "to the ends": [band(300.0, 500.0)],
    "nothing": [band(900.0, 901.0)],
    "two surfaces": [band(450.0, 600.0), band(550.0, 690.0, n_theta=2)],
    "disjoint": [band(450.0, 500.0), band(550.0, 690.0)],
    "everything": [band(0.0, 2000.0, T=1.0)],
}


@pytest.mark.parametrize("precision", [P.PLAIN_FP64, P.MIXED, P.MIXED_DS])
@pytest.mark.parametrize("name", COATINGS)
def test_interval_matches_the_test_by_wavelength(name, precision):
    counts = [20000, 333, 0, 4097, 12001]
    sc = G.test_system_scene(sources=G.mixed_sources(counts, seed=4), atmosphere=False)
    sc.coatings = list(COATINGS[name])
    sc.surfaces[4].coating = 1 if len(sc.coatings) > 1 else -1
    sc.sources.bundle = np.array([1, 1, 1, 8, 1], np.int32)
    sc.sources.bundle_sigma = np.full(5, 0.01)
    draw = G.run_gpu(sc, precision, records=False, early_reject=True)
    lam = G.run_gpu(sc, precision, records=True, early_reject=True)
    off = G.run_gpu(sc, precision, records=False, early_reject=False)
    assert np.array_equal(draw["image"], lam["image"]) and np.array_equal(draw["image"], off["image"])
    assert np.array_equal(draw["counters"], lam["counters"])
    assert (name in ("nothing", "disjoint")) == (int(draw["counters"][1]) == 0)
    np.testing.assert_allclose(draw["moments"], lam["moments"], rtol=1e-9, atol=1e-12)

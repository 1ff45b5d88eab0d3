"""The FP64 optics on surface shapes around the rules of its intersection: the single-precision start, its FP64
fallback for grazing rays, the sphere's and the conic's normals, even, odd and Zernike terms alone and together,
flat surfaces, tilts and decenters; the trace against the oracle's records and the adjoint against its dual numbers.

Tolerances.  Positions: both sides resolve an intersection to 1e-8 mm; over a radius of 40 mm and a path of 500 mm
that is 1.3e-7 mm at the detector from each, within the 1e-6 mm (1e-5 of the 0.1 mm pixel) asked for.  Rays that
graze the sphere of 24 mm lose digits without bound, so there one in a thousand may be off.  Gradients: both are
exact derivatives evaluated in FP64, 1e-6 of each parameter's scale as in test_gpu_grad."""
import ctypes as C

import numpy as np
import pytest

from paper_1504_06570_gb300 import inputs as I
from paper_1504_06570_gb300 import phosim as P
from tests import gpu_helpers as G
from tests.test_gpu_grad import oracle_gradient

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]

P_MISSED = 2               # PHOSIM_LOST_MISSED
ZERN = (0.0, 1e-5, -2e-5, 3e-5, 2e-5, -1e-5, 1e-5, 4e-6, 0.0, 2e-6, 5e-6, 0.0, 0.0, 1e-6, 0.0, 2e-6, 1e-6, 0.0, 0.0,
        3e-6, 1e-6, 2e-6, 0.0, 1e-6, 0.0, 0.0, 2e-6, 1e-6)
LENSES = {
    "sphere": dict(R=900.0),
    "steep sphere": dict(R=40.0),
    "grazed sphere": dict(R=24.0),
    "weak sphere": dict(R=1e7),
    "hyperboloid": dict(R=300.0, kappa=-5.0),
    "oblate": dict(R=-200.0, kappa=3.0),
    "paraboloid": dict(R=250.0, kappa=-1.0),
    "even": dict(R=5000.0, kappa=-0.5, alpha=(0, 2e-9, 0, 1e-13, 0, -1e-17, 0, 1e-21)),
    "odd": dict(alpha=(1e-7, 0, 1e-10, 0, -1e-14, 0, 1e-18, 0)),
    "even and odd": dict(R=700.0, kappa=0.4, alpha=(1e-7, 2e-9, 1e-11, 1e-13, 0, 0, 1e-19, 0)),
    "figure on a flat": dict(zern=ZERN, zern_rnorm=60.0),
    "figure, tilt and decenter": dict(R=900.0, kappa=-0.3, alpha=(0, 1e-9, 0, 0, 0, 0, 0, 0), zern=ZERN, zern_rnorm=60.0,
                                      pert=(0.3, -0.2, 0.1, 2e-3, -1e-3, 3e-2)),
}


def lens_scene(lens, n=20000):
    mats = [I.Material(I.VACUUM), I.Material(I.SELLMEIER, I.FUSED_SILICA_B, I.FUSED_SILICA_C), I.Material(I.SILICON)]
    surfaces = [I.Surface(kind=I.MIRROR, R=20000.0, kappa=-1.0, z=0.0, r_in=0.0, r_out=500.0),
                I.Surface(kind=I.REFRACT, z=9500.0, r_out=60.0, material=1, **lens),
                I.Surface(kind=I.REFRACT, z=9540.0, r_out=60.0, material=0, zern_rnorm=60.0, pert=(0.1, 0.0, 0.0, 1e-3, 2e-3, 0.0)),
                I.Surface(kind=I.DETECTOR, z=10007.5, material=2, pert=(0.0, 0.0, 0.0, 1e-3, 0.0, 0.0))]
    det = I.Detector(nx=700, ny=701, pixel=0.1, t_si=0.1, ell_lam0=400.0, ell_dlam=1.0,
                     ell=I.absorption_length_table(400.0, 1.0, 301), sigma=np.array([0.003, 0.003]))
    return I.Scene(seed=3, pupil_r_in=0.0, pupil_r_out=500.0, surfaces=surfaces, materials=mats, coatings=[], detector=det,
                   layers=[], sed_lam0=400.0, sed_dlam=1.0, sed_flux=I.sed_tables([5800.0], 400.0, 1.0, 300),
                   sersic=np.ones((1, 4)), sources=I.point_sources([0.0, 3e-5], [1e-5, -4e-5], [n, n // 3]),
                   atmosphere=False, sensor=False)


@pytest.mark.parametrize("precision", [P.PLAIN_FP64, P.MIXED])
@pytest.mark.parametrize("name", LENSES)
def test_records_match_oracle(oracle_mod, name, precision):
    sc = lens_scene(LENSES[name])
    gpu = G.run_gpu(sc, precision, moments=False)
    ora = G.oracle_trace(oracle_mod, sc)
    assert np.any(ora["flags"] & 1)
    if name == "grazed sphere":
        # the oracle's first guess is the paraboloid, and it drops a ray whose guess lies beyond the sphere's rim (missed
        # at surface 1) though the ray meets the sphere: those rays have no value to compare with
        known = ora["flags"] != ((P_MISSED << 8) | (1 << 16))
        gpu["rec"], ora = gpu["rec"][known], {k: v[known] if np.ndim(v) == 1 else v for k, v in ora.items()}
    G.compare_records(sc, gpu, ora, pos_tol_px=1e-5, min_frac=0.999 if name == "grazed sphere" else 1.0)


@pytest.mark.parametrize("name", ["steep sphere", "hyperboloid", "even and odd", "figure on a flat", "figure, tilt and decenter"])
def test_adjoint_matches_oracle(oracle_mod, name):
    sc = lens_scene(LENSES[name], n=900)
    sc.surfaces[1].zern_rnorm = 60.0
    sc.sensor = name != "steep sphere"
    params = [(s, f) for s in range(4) for f in (5, 0, 3, 1, 4, 2)] + [(1, 100 + j) for j in range(28)] + \
        [(2, 103), (2, 127), (2, 100)]
    dL = np.random.default_rng(1).normal(size=(2, 5))
    s = P.Scene(sc, P.PLAIN_FP64)
    g, _ = s.grad(dL, params)
    few, _ = s.grad(dL, params[30:33])              # a single surface: the sweep ends there
    s.close()
    go = oracle_gradient(oracle_mod, sc, dL, params)
    scale = np.abs(go).max(axis=0)
    scale = np.where(scale > 1e-9 * scale.max(), scale, scale.max())    # a derivative that vanishes by symmetry
    assert np.max(np.abs(g - go) / scale) < 1e-6
    np.testing.assert_allclose(few, g[:, 30:33], rtol=1e-12)


def fp64_eval(op, a):
    a = np.ascontiguousarray(a, np.float64)
    out, dp = np.zeros(len(a)), C.POINTER(C.c_double)
    assert P.lib().phosim_fp64_eval(op, a.ctypes.data_as(dp), out.ctypes.data_as(dp), len(a)) == 0
    return out


def test_fp64_helpers():
    """Reciprocal and roots: two roundings and a truncation near 2^-57 leave less than 2^-52, and the reference rounds
    once more (2^-53), so 2^-51 of the value; the conversions and the floor are exact."""
    rng = np.random.default_rng(3)
    v = 10.0 ** rng.uniform(-30, 30, 20000) * rng.uniform(1.0, 2.0, 20000)
    s = v * rng.choice([-1.0, 1.0], v.size)
    for op, x, ref in ((0, s, 1.0 / s), (1, v, 1.0 / np.sqrt(v)), (2, v, np.sqrt(v))):
        assert np.max(np.abs(fp64_eval(op, x) / ref - 1.0)) < 2.0 ** -51
    assert fp64_eval(2, [0.0])[0] == 0.0
    t = fp64_eval(3, s)
    assert np.array_equal(t, t.astype(np.float32)) and np.all(np.abs(t) <= np.abs(s)) and np.all(np.abs(t - s) < 2.0 ** -23 * np.abs(s))
    unit = np.r_[0.0, rng.random(20000), 1.0 - 2.0 ** -np.arange(20.0, 53.0), 2.0 ** -np.arange(1.0, 50.0), 0.5 + 2.0 ** -25,
                 0.5 + 3 * 2.0 ** -25]
    assert np.array_equal(fp64_eval(4, unit), unit.astype(np.float32).astype(np.float64))
    f = np.r_[0.0, s].astype(np.float32).astype(np.float64)
    assert np.array_equal(fp64_eval(5, f), f)
    x = np.r_[rng.uniform(-2.0 ** 31, 2.0 ** 31, 20000) * 10.0 ** rng.uniform(-9, 0, 20000), 0.0, -0.0, 1.0, -1.0, -1e-300, 2.0 ** 31 - 1]
    assert np.array_equal(fp64_eval(6, x), np.floor(x)) and np.array_equal(fp64_eval(7, x), np.floor(x))
    w = np.r_[0.0, 1.0, 2.0 ** 32 - 1, rng.integers(0, 2 ** 32, 1000).astype(np.float64)]
    assert np.array_equal(fp64_eval(8, w), (w + 0.5) * 2.0 ** -32)

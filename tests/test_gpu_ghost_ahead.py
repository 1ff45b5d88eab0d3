"""A ghost meets only surfaces ahead of it, also where the next surface is a few 1e-7 mm away and steep: a ray that a
coating turns round in a bowl goes back through an uncoated one of the same shape just above, then out through a flat.  The
distance is far below the rounding of the single-precision start of the intersection (1e-6 mm at 5 mm from the vertex
plane), and far above that of the FP64 position (1e-15 mm).  Fates and places are the oracle's."""
import numpy as np
import pytest

from paper_1504_06570_gb300 import inputs as I
from paper_1504_06570_gb300 import phosim as P
from tests import gpu_helpers as G
from tests import helpers as H

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


@pytest.mark.parametrize("precision", [P.PLAIN_FP64, P.MIXED])
@pytest.mark.parametrize("gap", [3e-7, 2e-6, 1e-3])
@pytest.mark.parametrize("shape", [dict(R=40.0), dict(R=40.0, kappa=-0.6), dict(R=-40.0)])
def test_surface_just_ahead(oracle_mod, shape, gap, precision):
    mats = [I.Material(I.VACUUM), I.Material(I.SELLMEIER, I.FUSED_SILICA_B, I.FUSED_SILICA_C), I.Material(I.SILICON)]
    surfaces = [I.Surface(kind=I.REFRACT, z=20.0, r_out=1000.0, material=0),
                I.Surface(kind=I.REFRACT, z=0.0, r_out=30.0, material=1, **shape),
                I.Surface(kind=I.REFRACT, z=-gap, r_out=30.0, material=0, coating=0, **shape),
                I.Surface(kind=I.DETECTOR, z=-40.0, material=2)]
    coat = I.Coating(lam0=400.0, dlam=300.0, theta0=0.0, dtheta=1.6, table=np.array([[0.3]]), reflect=np.array([[0.6]]))
    sc = H.bare_scene(surfaces, materials=mats, coatings=[coat], nx=300, pixel=0.5, n_photons=5000, pupil=(14.0, 22.0))
    gpu = G.run_gpu(sc, precision, moments=False)
    ora = G.oracle_trace(oracle_mod, sc)
    missed_above = (2 << 8) | (0 << 16)          # gone back past the first surface
    assert np.sum(ora["flags"] == missed_above) > 2000
    G.compare_records(sc, gpu, ora, pos_tol_px=1e-5)

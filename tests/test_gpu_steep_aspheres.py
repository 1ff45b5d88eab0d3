"""Aspheres whose terms are steep past their edge, met by rays that come in outside the aperture or at a slant: Newton's method
from the conic's root does not settle on them, or leaves the conic's domain, and that is their fate (the oracle's: not
converged, or missed), whatever other crossing a faster iteration would come to.  Fates of every photon, and the places of
those detected (within 1e-5 of the pixel, as test_gpu_fp64_surfaces), in the two FP64 precisions."""
import numpy as np
import pytest

from paper_1504_06570_gb300 import inputs as I
from paper_1504_06570_gb300 import phosim as P
from tests import gpu_helpers as G
from tests import helpers as H

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


def terms(r, **edge):
    """alpha_3 .. alpha_10 from the sag of each term (mm) at radius r."""
    a = [0.0] * 8
    for name, sag in edge.items():
        k = int(name[1:])
        a[k - 3] = sag / float(r) ** k
    return tuple(a)


SYSTEMS = {
    # a mirror with 0.7 mm of a seventh-order term throws its outer rays past the lens's rim
    "thrown past a lens": ([
        I.Surface(kind=I.MIRROR, R=20730.0, z=0.0, r_out=500.0, alpha=terms(500, a3=0.063, a4=0.11, a7=0.67)),
        I.Surface(kind=I.REFRACT, R=779.0, kappa=-1.0, z=9405.0, r_out=60.0, material=1, alpha=terms(60, a5=0.24, a10=0.17)),
        I.Surface(kind=I.REFRACT, R=19380.0, kappa=-0.7, z=9446.0, r_out=60.0, material=0)], 10009.0, (0.0, 500.0), 0.05, 7e-5),
    # lenses with high terms, rays up to 30 degrees off the axis
    "slanting rays": ([
        I.Surface(kind=I.REFRACT, R=41250.0, kappa=-1.0, z=0.0, r_out=40.0, material=1),
        I.Surface(kind=I.REFRACT, z=-193.0, r_out=40.0, material=0, alpha=terms(40, a9=-0.12)),
        I.Surface(kind=I.REFRACT, R=6019.0, z=-202.0, r_out=40.0, material=1, alpha=terms(40, a7=-0.0063)),
        I.Surface(kind=I.REFRACT, R=1979.0, z=-219.7, r_out=40.0, material=0)], -419.0, (0.0, 25.0), 0.7, 0.5),
}


@pytest.mark.parametrize("precision", [P.PLAIN_FP64, P.MIXED])
@pytest.mark.parametrize("name", SYSTEMS)
def test_fates_are_newtons(oracle_mod, name, precision):
    surfaces, z_det, pupil, pixel, field = SYSTEMS[name]
    mats = [I.Material(I.VACUUM), I.Material(I.SELLMEIER, I.FUSED_SILICA_B, I.FUSED_SILICA_C), I.Material(I.SILICON)]
    xi = np.linspace(-field, field, 8)
    sc = H.bare_scene(surfaces + [I.Surface(kind=I.DETECTOR, z=z_det, material=2)], materials=mats, nx=512, pixel=pixel, pupil=pupil,
                      sources=I.point_sources(xi, 0.8 * xi[::-1], [5000] * 8))
    gpu = G.run_gpu(sc, precision, moments=False)
    ora = G.oracle_trace(oracle_mod, sc)
    assert np.sum(ora["flags"] & 1) > 1000
    assert np.any((ora["flags"] >> 8 & 0xff) == 3)              # rays that do not settle are among them
    G.compare_records(sc, gpu, ora, pos_tol_px=1e-5)

"""Rays that meet a conic twice on its vertex branch: the crossing nearer to where the ray comes from counts (the oracle's
first guess is the paraboloid's root of the smaller distance, exact for these surfaces), whichever of the two is nearer to
the plane of the vertex.  Sources 20 to 65 degrees off the axis of deep paraboloids, with and without an even term, against
the oracle's fates and places.  The two crossings are more than 20 mm apart; the places are asked for to 0.5 mm, which
leaves room for what rays that come in along the bowl's side lose of the 1e7 mm of their path to it (0.06 mm in
double-single, whose positions carry some 2^-45 of that)."""
import numpy as np
import pytest

from paper_1504_06570_gb300 import inputs as I
from paper_1504_06570_gb300 import phosim as P
from tests import gpu_helpers as G
from tests import helpers as H

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


@pytest.mark.parametrize("precision", [P.PLAIN_FP64, P.MIXED, P.MIXED_DS])
@pytest.mark.parametrize("R, r_out, alpha", [(40.0, 500.0, ()), (40.0, 60.0, ()), (-40.0, 500.0, ()), (90.0, 500.0, (0.0, 1e-10))])
def test_first_crossing_counts(oracle_mod, R, r_out, alpha, precision):
    mats = [I.Material(I.VACUUM), I.Material(I.SELLMEIER, I.FUSED_SILICA_B, I.FUSED_SILICA_C), I.Material(I.SILICON)]
    a = tuple(alpha) + (0.0,) * (8 - len(alpha))
    surfaces = [I.Surface(kind=I.REFRACT, R=R, kappa=-1.0, z=0.0, r_out=r_out, material=1, alpha=a),
                I.Surface(kind=I.DETECTOR, z=-40.0, material=2)]
    sc = H.bare_scene(surfaces, materials=mats, nx=400, pixel=5.0, pupil=(0.0, 30.0),
                      sources=I.point_sources([0.35, 0.5, -0.7, 0.2, 0.9], [0.0, 0.2, 0.1, -0.4, 0.0], [2000] * 5))
    rec = G.run_gpu(sc, precision, moments=False)["rec"]
    ora = G.oracle_trace(oracle_mod, sc)
    assert np.sum(ora["flags"] & 1) > 500
    assert np.all((rec["flags"] == ora["flags"]) | G.boundary_mask(ora))
    both = ((rec["flags"] & 1) & (ora["flags"] & 1)) == 1
    for c in ("x", "y"):
        assert np.max(np.abs(rec[c][both] - ora[c][both])) < 0.5

"""The detector's steps of the FP64 paths against the oracle's records: table lookups off either end of the absorption
lengths, the chip's edges, the dead layer (0, -0 and a fifth of the thickness) and the back side, and coatings of one angle
bin, decided in the dynamic transmission test alone, and of two.  The oracle and the FP64 path take the same decisions on
the same draws except within a rounding of an edge, so every fate is the same but for one in 1e5, and positions agree to
1e-4 of a pixel."""
import numpy as np
import pytest

from paper_1504_06570_gb300 import inputs as I
from paper_1504_06570_gb300 import phosim as P
from tests import gpu_helpers as G

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


@pytest.mark.parametrize("dead_layer, angles, chip", [(0.0, 1, 512), (-0.0, 2, 64), (0.02, 1, 33), (0.02, 2, 512)])
@pytest.mark.parametrize("early", [False, True])
def test_detector_matches_oracle(oracle_mod, dead_layer, angles, chip, early):
    sc = G.test_system_scene(n_photons=30000, atmosphere=False, chip=chip)
    d = sc.detector
    d.ell_lam0, d.ell = 520.0, I.absorption_length_table(520.0, 1.0, 61)
    d.dead_layer = dead_layer
    table = np.repeat(np.where(np.arange(300) % 7 < 5, 0.9, 0.1)[:, None], angles, 1)
    if angles == 2:
        table[:, 1] *= 0.5
    sc.coatings = [I.Coating(lam0=400.0, dlam=1.0, theta0=0.0, dtheta=0.005, table=table.copy())]
    gpu = G.run_gpu(sc, P.PLAIN_FP64, moments=False, early_reject=early)
    ora = G.oracle_trace(oracle_mod, sc)
    assert int((ora["flags"] & 1).sum()) < 30000   # (none reach the chip of 33 pixels, in the defocused ring's hole)
    if early:                                     # the same fates in another order: the detected photons are the same
        g, o = gpu["rec"], ora
        both = ((g["flags"] & 1) == 1) & ((o["flags"] & 1) == 1)
        assert np.sum((g["flags"] & 1) != (o["flags"] & 1)) <= 1
        assert np.all(np.abs(g["x"][both] - o["x"][both]) < 1e-4 * d.pixel)
    else:
        G.compare_records(sc, gpu, ora)

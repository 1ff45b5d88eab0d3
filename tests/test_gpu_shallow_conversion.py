"""Conversion draws at the top of the 32-bit range, which round to 1 in single precision: a conversion length of zero (its
logarithm negated, -0).  The photon converts at the sensor's surface and is detected there, as the oracle's, whose length
is below 1e-9 of the absorption length.  The three photons with such a draw are those below 6e8 of source 0 with seed
12345, found by running the generator."""

import numpy as np
import pytest

from paper_1504_06570_gb300 import phosim as P
from tests import gpu_helpers as G

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


@pytest.mark.parametrize("precision", [P.PLAIN_FP64, P.MIXED, P.MIXED_DS])
@pytest.mark.parametrize("early", [False, True])
def test_length_of_zero(oracle_mod, precision, early):
    sc = G.test_system_scene(n_photons=1, atmosphere=False)
    assert sc.seed == 12345
    detected = 0
    for photon in (530445959, 593783117, 598834038):
        n, first = np.array([1], np.uint64), np.array([photon], np.uint64)
        rec = G.run_gpu(sc, precision, moments=False, n_photons=n, first=first, early_reject=early)["rec"]
        ora = G.oracle_trace(oracle_mod, sc, n_photons=n, first=first)
        assert (int(rec["flags"][0]) & 1) == (int(ora["flags"][0]) & 1), (photon, hex(int(rec["flags"][0])), hex(int(ora["flags"][0])))
        assert (int(rec["flags"][0]) >> 8) & 0xff != 7               # PHOSIM_LOST_NOT_CONVERTED
        if int(rec["flags"][0]) & 1:
            detected += 1
            assert abs(rec["x"][0] - ora["x"][0]) < 1e-2 * sc.detector.pixel
            assert abs(rec["y"][0] - ora["y"][0]) < 1e-2 * sc.detector.pixel
    assert detected >= 1

"""The launch counters after a gradient are those of its forward pass, also where the adjoint makes the photon batches
again: without a coated surface, and with more photons than one chunk of batches (2^27).  Every photon is traced once and
ends once."""
import numpy as np
import pytest

from paper_1504_06570_gb300 import inputs as I
from paper_1504_06570_gb300 import phosim as P
from tests import gpu_helpers as G

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


@pytest.mark.parametrize("counts, coated", [([5000, 0, 33], True), ([5000, 0, 33], False), ([1], False), ([2 ** 27 + 300000], True)])
def test_photons_counted_once(counts, coated):
    sc = G.test_system_scene(sources=G.mixed_sources(counts, seed=6), atmosphere=False)
    sc.coatings = [I.Coating(lam0=400.0, dlam=300.0, theta0=0.0, dtheta=1.6, table=np.array([[0.05 if sum(counts) > 10 ** 6 else 0.7]]))]
    if not coated:
        sc.surfaces[3].coating = -1
    s = P.Scene(sc, P.PLAIN_FP64, early_reject=True)
    img = torch.zeros((sc.detector.ny, sc.detector.nx), dtype=torch.int32, device="cuda")
    s.trace(img)
    traced = s.counters()
    s.grad(np.ones((len(counts), 5)), [(1, 0), (5, 2)])
    after = s.counters()
    s.close()
    assert int(after[0]) == sum(counts) and int(after.sum()) == 2 * sum(counts)
    assert np.array_equal(after, traced)

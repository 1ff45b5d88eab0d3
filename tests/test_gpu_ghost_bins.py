"""Ghost rounds with rays of several coated surfaces in one round, placed by blocks of 2048 rays: plates that pass part of
the light, so that the first round holds rays turned at each of three surfaces and further rounds those turned again.  The
photon counts put the first round's population (about 0.63, 0.19 and 0.06 of the photons, from the three plates) around
one and several blocks.  Records, image and counts are those of the one-kernel path."""
import numpy as np
import pytest

from paper_1504_06570_gb300 import phosim as P
from tests import gpu_helpers as G
from tests.test_gpu_ghost_rounds import ghost_scene, one_kernel

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]

LOST_COATING = 5


@pytest.mark.parametrize("photons", [40, 2320, 2330, 2340, 4650, 4660, 4670, 20481, 700001])
def test_rays_of_three_surfaces_have_one_place_each(photons):
    sc = ghost_scene([photons], 0.7, 1)
    two, one = G.run_gpu(sc, P.MIXED_DS, early_reject=False), one_kernel(sc, False)
    assert np.array_equal(two["rec"], one["rec"]) and np.array_equal(two["image"], one["image"])
    assert int(two["counters"][0]) == photons and int(two["counters"].sum()) == 2 * photons
    if photons > 2000:
        rec = two["rec"]
        reason, surface = (rec["flags"] >> 8) & 0xff, rec["flags"] >> 16
        # absorbed at each plate (so each plate was reached, and turns nine rays for each one that it absorbs), and detected
        assert {1, 2, 4} <= set(surface[reason == LOST_COATING]) and int(two["image"].sum()) > 0

"""The order of a round's rays, which blocks of 2048 rays place together: every ray is walked once, so the records, the image
and the counts are those of the one-kernel path.  Nearly every ray is turned at its first coated plate, so that a round holds
about as many rays as reach it: from none, by one and a few, to those around one and several blocks' worth, from one surface
and from three."""
import numpy as np
import pytest

from paper_1504_06570_gb300 import phosim as P
from tests import gpu_helpers as G
from tests.test_gpu_ghost_rounds import ghost_scene, one_kernel

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


@pytest.mark.parametrize("surfaces", [(1,), (1, 2, 4)])
@pytest.mark.parametrize("photons", [1, 33, 2047, 2048, 2049, 2300, 4096, 4600, 20481, 700001])
def test_every_ray_has_one_place(photons, surfaces):
    sc = ghost_scene([photons], 1.0, 1)
    for k in (1, 2, 4):
        sc.surfaces[k].coating = 1 if k in surfaces else -1
    two, one = G.run_gpu(sc, P.MIXED_DS, early_reject=False), one_kernel(sc, False)
    assert np.array_equal(two["image"], one["image"]) and np.array_equal(two["rec"], one["rec"])
    assert int(two["counters"][0]) == photons and int(two["counters"].sum()) == 2 * photons

"""Host images around the rule that adds only a short exposure's pixels with counts to a pinned image: the counts added to
what the image held are those of a device image, for pinned and pageable memory, below, at and above the size where the
image is staged instead (a photon that may pass for every twelfth pixel), in every precision, twice in a row."""
import numpy as np
import pytest

from paper_1504_06570_gb300 import phosim as P
from tests import gpu_helpers as G
from tests.test_gpu_pass_draws import band

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


@pytest.mark.parametrize("precision", [P.PLAIN_FP64, P.MIXED, P.MIXED_DS])
@pytest.mark.parametrize("pinned", [True, False])
@pytest.mark.parametrize("photons, coating", [(3, None), (2730, None), (2731, None), (40000, None), (5000, "half"), (6000, "half"),
                                              (2047, "shut")])
def test_host_image_is_the_device_image(precision, pinned, photons, coating):
    sc = G.test_system_scene(sources=G.mixed_sources([photons], seed=6), chip=181)         # 32761 pixels: 2730.08 photons
    sc.coatings = [band(0.0, 2000.0, T=0.9) if coating is None else band(400.0, 550.0) if coating == "half" else band(900.0, 901.0)]
    d = sc.detector
    s = P.Scene(sc, precision, early_reject=True)
    dev = torch.zeros((d.ny, d.nx), dtype=torch.int32, device="cuda")
    s.trace(dev)
    old = torch.from_numpy(np.random.default_rng(1).integers(0, 2 ** 31, (d.ny, d.nx)).astype(np.int32))
    img = old.clone().pin_memory() if pinned else old.clone()
    for k in (1, 2):
        s.trace(img)                          # returns with the counts in the host's memory
        assert torch.equal(img, (old.long() + k * dev.cpu().long()).to(torch.int32))
    s.close()

"""Saturation and bleeding (Sec. 2.5): the warp-per-half-row kernel against the oracle at the sizes where it can go
wrong: half-rows around one warp, one batch of loads and one chunk of distances, odd widths (halves of different
lengths), the widest half-row that is worked in shared memory and one worked in place, and full wells from zero to
the largest count.  Whole numbers: equal."""
import numpy as np
import pytest

from paper_1504_06570_gb300 import phosim as P

pytestmark = pytest.mark.gpu


def crowded(nx, ny, well, fill, seed):
    """Sky around a fraction of the full well, with peaks that `fill` times the room of the image would take."""
    rng = np.random.default_rng(seed)
    sky = rng.integers(0, max(1, min(well, 2 ** 31)) + 1, (ny, nx)).astype(np.uint64)
    peaks = rng.random((ny, nx)) < rng.choice([0.002, 0.05, 0.4], (ny, 1))
    room = float(np.maximum(0.0, well - sky.astype(np.float64)).sum())
    each = fill * room / max(1, int(peaks.sum()))
    sky[peaks] += rng.integers(0, int(min(2 * each + 2, 2 ** 31)), int(peaks.sum())).astype(np.uint64)
    return np.minimum(sky, 2 ** 32 - 1).astype(np.uint32)


@pytest.mark.parametrize("nx, ny", [(2, 1), (3, 2), (63, 5), (64, 9), (65, 3), (129, 4), (511, 7), (514, 33), (1023, 6),
                                    (4096, 12), (24570, 3), (24571, 2)])
@pytest.mark.parametrize("well, fill", [(0, 0.5), (1, 0.3), (1000, 0.05), (1000, 0.9), (1000, 3.0), (2 ** 32 - 1, 0.5)])
def test_bleed_matches_oracle(oracle_mod, nx, ny, well, fill):
    import torch
    img = crowded(nx, ny, well, fill, 7 * nx + ny)
    t = torch.from_numpy(img.view(np.int32).copy()).cuda()
    removed = P.bleed(t, well)
    ref, ref_removed = oracle_mod.bleed(img, well)
    assert np.array_equal(t.cpu().numpy().view(np.uint32), ref)
    assert int(removed.item()) == ref_removed

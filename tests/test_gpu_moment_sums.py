"""The moment sums of the double-single path: a warp with up to 8 runs of one source sums each run before its atomics, one
with more adds every photon.  Sources of one photon to whole warps and more, so that warps hold one run, the limit and
more, with bundles (whose photons are summed a ray at a time), above and below the size where the sums are striped: the
sums over the records about the chief rays.  The tolerance is two roundings of a single-precision offset, 2^-22 of the
sum of the terms' sizes (a record's offset from the chief ray may round the other way); a photon left out or counted twice
is off by at least 1 / 70000 of it."""
import numpy as np
import pytest

from paper_1504_06570_gb300 import phosim as P
from tests import gpu_helpers as G

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


@pytest.mark.parametrize("bundle", [1, 5])
@pytest.mark.parametrize("counts", [[1] * 300, [1, 2, 3] * 100, [5] * 64, [4, 40, 4, 4] * 50, [33, 31, 64, 1, 70] * 9,
                                    [30000, 7, 39000, 1, 1, 1, 1, 1, 1, 1, 1, 1, 64], [70000]])
def test_sums_are_those_of_the_records(counts, bundle):
    sc = G.test_system_scene(sources=G.mixed_sources(counts, seed=7))
    sc.sources.bundle = np.full(len(counts), bundle, np.int32)
    sc.sources.bundle_sigma = np.full(len(counts), 0.01)
    s = P.Scene(sc, P.MIXED_DS, early_reject=False)
    d = sc.detector
    img = torch.zeros((d.ny, d.nx), dtype=torch.int32, device="cuda")
    rec = torch.zeros(sum(counts) * P.RECORD_DTYPE.itemsize, dtype=torch.uint8, device="cuda")
    mom = torch.zeros((len(counts), P.MOMENT_WORDS), dtype=torch.float64, device="cuda")
    s.trace(img, rec, mom)
    r, m, ends = P.records_to_numpy(rec), mom.cpu().numpy(), np.cumsum(counts)
    counters = s.counters()
    s.close()
    hit = (r["flags"] & 1) == 1
    pix = np.bincount(r["pix"][hit], minlength=d.nx * d.ny).reshape(d.ny, d.nx)
    assert np.array_equal(img.cpu().numpy(), pix) and int(counters[1]) == int(hit.sum()) > 0
    for k, n in enumerate(counts):
        q = r[ends[k] - n:ends[k]]
        q = q[(q["flags"] & 1) == 1]
        dx, dy = ((q[c] - m[k, j]).astype(np.float32).astype(np.float64) for c, j in (("x", 6), ("y", 7)))
        terms = [np.ones(len(q)), dx, dy, dx * dx, dx * dy, dy * dy]
        ref, scale = (np.array([f(t).sum() for t in terms]) for f in (lambda t: t, np.abs))
        assert m[k, 0] == len(q)
        assert np.all(np.abs(m[k, :6] - ref) <= 2.0 ** -22 * scale), (counts[:5], k, m[k], ref)

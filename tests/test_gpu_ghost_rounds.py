"""Ghosts of the two-kernel double-single path, whose turned rays leave their block and are walked in rounds: the same
records, images and counts as the one-kernel path (phosim_trace_noalloc), which walks every ray in place.  Same
arithmetic per ray, so whole numbers and positions are equal and the moment sums agree to their summation order.
Sizes: fewer rays than a block, blocks with a remainder, more rays than one chunk (2^24 with reflecting coatings), few
and many reflections a ray (more than the rounds), bundles, and the call as one graph."""
import ctypes as C

import numpy as np
import pytest

from paper_1504_06570_gb300 import inputs as I
from paper_1504_06570_gb300 import phosim as P
from tests import gpu_helpers as G

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


def ghost_scene(counts, reflect, bundle):
    sc = G.test_system_scene(sources=G.mixed_sources(counts, seed=2), chip=301)
    lam = np.zeros((300, 2))
    plate = I.Coating(lam0=400.0, dlam=1.0, theta0=0.0, dtheta=0.01, table=lam + (1.0 - reflect), reflect=lam + 0.9 * reflect)
    sc.coatings.append(plate)
    for k in (1, 2, 4):
        sc.surfaces[k].coating = 1
    if bundle > 1:
        sc.sources.bundle = np.where(np.arange(len(counts)) % 2 == 0, bundle, 1).astype(np.int32)
        sc.sources.bundle_sigma = np.full(len(counts), 0.02)
    return sc


def one_kernel(sc, early):
    s = P.Scene(sc, P.MIXED_DS, early_reject=early)
    L = s.L
    L.phosim_trace_noalloc.argtypes = [C.c_void_p, C.POINTER(P.Source), C.c_int, C.POINTER(C.c_uint64),
                                       C.POINTER(C.c_uint64), C.c_void_p, C.c_void_p, C.c_void_p, C.c_void_p]
    n, d = int(sc.sources.n_photons.sum()), sc.detector
    img = torch.zeros((d.ny, d.nx), dtype=torch.int32, device="cuda")
    rec = torch.zeros(n * P.RECORD_DTYPE.itemsize, dtype=torch.uint8, device="cuda") if n < 10 ** 6 else None
    mom = torch.zeros((len(sc.sources), P.MOMENT_WORDS), dtype=torch.float64, device="cuda")
    rc = L.phosim_trace_noalloc(s.h, s.src, len(sc.sources), s.n_photons.ctypes.data_as(C.POINTER(C.c_uint64)), None,
                                C.c_void_p(img.data_ptr()), C.c_void_p(rec.data_ptr()) if rec is not None else None,
                                C.c_void_p(mom.data_ptr()), C.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == 0
    torch.cuda.synchronize()
    s.close()
    return {"image": img.cpu().numpy().view(np.uint32), "rec": None if rec is None else P.records_to_numpy(rec),
            "moments": mom.cpu().numpy()}


@pytest.mark.parametrize("counts, reflect, bundle, early, graph", [
    ([7], 0.5, 1, False, False),
    ([255, 258, 1, 0, 4097], 0.7, 1, False, True),
    ([30001, 20011, 5], 0.95, 1, True, False),
    ([3000, 4000, 5003], 0.6, 7, False, True),
    ([9_000_001, 9_000_000], 0.3, 1, False, True),
    ([9_000_001, 9_000_000], 0.3, 1, False, False)])
def test_rounds_match_the_walk_in_place(counts, reflect, bundle, early, graph):
    sc = ghost_scene(counts, reflect, bundle)
    records = sum(counts) < 10 ** 6
    two = G.run_gpu(sc, P.MIXED_DS, records=records, early_reject=early, graph=graph)
    one = one_kernel(sc, early)
    assert np.array_equal(two["image"], one["image"])
    assert int(two["counters"][0]) == sum(counts) and int(two["counters"].sum()) == 2 * sum(counts)
    np.testing.assert_allclose(two["moments"], one["moments"], rtol=1e-6, atol=1e-9)
    if records:
        assert np.array_equal(two["rec"], one["rec"])

"""The FP64 paths with the dynamic transmission test (batches of photons that go on, a warp a batch) against the
one-kernel path of phosim_trace_noalloc: the same records, images, counts and, to the order of their sums, moments.
Sizes: batches with one photon, full ones and remainders, tiles of one warp and long ones, empty sources, bundles,
scenes whose coatings stop nothing or everything, a call as a graph, and more photons than one chunk (2^27).  The adjoint
takes the trace's batches, or makes them again where they came in chunks: against central differences as in
test_gpu_grad."""
import ctypes as C

import numpy as np
import pytest

from paper_1504_06570_gb300 import phosim as P
from tests import gpu_helpers as G
from tests.test_gpu_pass_draws import band

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


def run(sc, precision, one_kernel, records, graph=False, tile=0):
    s = P.Scene(sc, precision, early_reject=True, graph=graph)
    if tile:
        s.set_schedule(128, tile)
    n, d = sc.sources.n_photons, sc.detector
    img = torch.zeros((d.ny, d.nx), dtype=torch.int32, device="cuda")
    rec = torch.zeros(max(1, int(n.sum())) * P.RECORD_DTYPE.itemsize, dtype=torch.uint8, device="cuda") if records else None
    mom = torch.zeros((len(n), P.MOMENT_WORDS), dtype=torch.float64, device="cuda")
    counters = None
    if one_kernel:
        L = s.L
        L.phosim_trace_noalloc.argtypes = [C.c_void_p, C.POINTER(P.Source), C.c_int, C.POINTER(C.c_uint64),
                                           C.POINTER(C.c_uint64), C.c_void_p, C.c_void_p, C.c_void_p, C.c_void_p]
        rc = L.phosim_trace_noalloc(s.h, s.src, len(n), s.n_photons.ctypes.data_as(C.POINTER(C.c_uint64)), None,
                                    C.c_void_p(img.data_ptr()), C.c_void_p(rec.data_ptr()) if records else None,
                                    C.c_void_p(mom.data_ptr()), C.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert rc == 0
    else:
        s.trace(img, rec, mom)
        counters = s.counters()
    torch.cuda.synchronize()
    s.close()
    return img, (P.records_to_numpy(rec)[:int(n.sum())] if records else None), mom.cpu().numpy(), counters


@pytest.mark.parametrize("precision", [P.PLAIN_FP64, P.MIXED])
@pytest.mark.parametrize("counts, tile, coating, graph", [
    ([1], 0, "band", False), ([33, 0, 31, 64], 32, "band", False), ([257, 4095], 64, "open", True),
    ([20011, 5, 0, 3000], 0, "band", True), ([40000], 4096, "band", False), ([5000, 77], 0, "shut", False),
    ([3000, 900, 64], 0, "bundles", False)])
def test_batches_match_one_kernel(precision, counts, tile, coating, graph):
    sc = G.test_system_scene(sources=G.mixed_sources(counts, seed=9))
    if coating == "open":
        sc.coatings = [band(0.0, 2000.0, T=1.0)]
    if coating == "shut":
        sc.coatings = [band(900.0, 901.0)]
    if coating == "bundles":
        sc.sources.bundle = np.array([8, 1, 5], np.int32)
        sc.sources.bundle_sigma = np.full(3, 0.02)
    img, rec, mom, cnt = run(sc, precision, False, True, graph, tile)
    img1, rec1, mom1, _ = run(sc, precision, True, True)
    assert np.array_equal(rec, rec1) and torch.equal(img, img1)
    lost = np.bincount((rec["flags"] >> 8) & 0xff, minlength=9)[1:9]
    assert list(cnt) == [sum(counts), int((rec["flags"] & 1).sum()), *lost]
    np.testing.assert_allclose(mom, mom1, rtol=1e-9, atol=1e-9)
    img2, _, mom2, cnt2 = run(sc, precision, False, False, graph, tile)
    assert torch.equal(img, img2) and np.array_equal(cnt, cnt2)
    np.testing.assert_allclose(mom2, mom, rtol=1e-9, atol=1e-9)


@pytest.mark.parametrize("graph", [False, True])
def test_chunks_match_one_kernel(graph):
    sc = G.test_system_scene(sources=G.mixed_sources([(1 << 27) + 4097, 30000001], seed=9), atmosphere=False, sensor=False)
    img, _, mom, cnt = run(sc, P.PLAIN_FP64, False, False, graph)
    img1, _, mom1, _ = run(sc, P.PLAIN_FP64, True, False)
    assert torch.equal(img, img1) and int(cnt[0]) == int(sc.sources.n_photons.sum())
    np.testing.assert_allclose(mom, mom1, rtol=1e-9, atol=1e-6)


def test_adjoint_of_chunks_matches_central_differences():
    sc = G.test_system_scene(sources=G.mixed_sources([(1 << 27) + 100003], seed=9), atmosphere=False)
    dL = np.random.default_rng(2).normal(size=(1, 5))
    params, steps = [(0, 3), (1, 0), (0, 104)], [1e-7, 1e-3, 1e-7]
    s = P.Scene(sc, P.PLAIN_FP64)
    g, _ = s.grad(dL, params)
    for k, (p, h) in enumerate(zip(params, steps)):
        base = sc.surfaces[p[0]].pert[p[1]] if p[1] < 6 else sc.surfaces[p[0]].zern[p[1] - 100]
        v = []
        for sign in (1, -1):
            s.set_parameters([p], [base + sign * h])
            _, m = s.grad(np.zeros((1, 5)), [p])
            v.append(float((dL * m[:, 1:]).sum()))
        s.set_parameters([p], [base])
        assert abs((v[0] - v[1]) / (2 * h) - g[0, k]) <= 1e-3 * abs(g[0, k]), (p, v, g[0, k])
    s.close()

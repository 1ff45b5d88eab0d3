"""The first kernel of a trace call: few sources travel in its parameters (12 at most), more are copied; it clears the
call's scratch, and the rays start beside the chief rays.  Calls on one scene with growing and shrinking source lists
around that limit, kernel by kernel and as a graph: every call's records, image and counts are those of
phosim_trace_noalloc, which copies its lists and runs its kernels one after the other; and the moments are the sums
over the records about the chief rays, below and above the size where the double-single path adds them directly
(65536 photons).  The moment tolerance is that of sums of up to 7e4 terms in FP64 about a point, 1e-9 of the largest
term's size, and in the mixed path of compensated single-precision sums, 1e-6."""
import ctypes as C

import numpy as np
import pytest

from paper_1504_06570_gb300 import phosim as P
from tests import gpu_helpers as G

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


def outputs(sc, n):
    d = sc.detector
    return (torch.zeros((d.ny, d.nx), dtype=torch.int32, device="cuda"),
            torch.zeros(int(np.sum(n)) * P.RECORD_DTYPE.itemsize, dtype=torch.uint8, device="cuda"),
            torch.zeros((len(n), P.MOMENT_WORDS), dtype=torch.float64, device="cuda"))


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("precision, rtol", [(P.PLAIN_FP64, 1e-9), (P.MIXED, 1e-6), (P.MIXED_DS, 1e-9)])
def test_calls_of_changing_lists(precision, rtol, graph):
    lists = [[500], [70, 0, 900], [100] * 12, [100] * 13, [37] * 50, [65536], [40000, 25537], [3] * 12]
    sc = G.test_system_scene(sources=G.mixed_sources(lists[0], seed=3))
    s = P.Scene(sc, precision, early_reject=True, graph=graph)
    L = s.L
    L.phosim_trace_noalloc.argtypes = [C.c_void_p, C.POINTER(P.Source), C.c_int, C.POINTER(C.c_uint64),
                                       C.POINTER(C.c_uint64), C.c_void_p, C.c_void_p, C.c_void_p, C.c_void_p]
    for counts in lists:
        s.set_sources(G.mixed_sources(counts, seed=3))
        img, rec, mom = outputs(sc, counts)
        s.trace(img, rec, mom)
        img2, rec2, mom2 = outputs(sc, counts)
        rc = L.phosim_trace_noalloc(s.h, s.src, len(counts), s.n_photons.ctypes.data_as(C.POINTER(C.c_uint64)), None,
                                    C.c_void_p(img2.data_ptr()), C.c_void_p(rec2.data_ptr()), C.c_void_p(mom2.data_ptr()),
                                    C.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert rc == 0
        r = P.records_to_numpy(rec)
        assert np.array_equal(r, P.records_to_numpy(rec2))
        assert torch.equal(img, img2) and int(img.sum()) == int((r["flags"] & 1).sum())
        assert int(s.counters()[0]) == sum(counts)
        m, ends = mom.cpu().numpy(), np.cumsum(counts)
        assert np.array_equal(m[:, 6:], mom2.cpu().numpy()[:, 6:])
        for k, n in enumerate(counts):
            q = r[ends[k] - n:ends[k]]
            q = q[(q["flags"] & 1) == 1]
            dx, dy = q["x"] - m[k, 6], q["y"] - m[k, 7]
            if precision == P.MIXED_DS:          # it sums exact products of the single-precision offsets
                dx, dy = dx.astype(np.float32).astype(np.float64), dy.astype(np.float32).astype(np.float64)
            ref = [len(q), dx.sum(), dy.sum(), (dx * dx).sum(), (dx * dy).sum(), (dy * dy).sum()]
            scale = [1.0, np.abs(dx).sum(), np.abs(dy).sum(), ref[3], np.abs(dx * dy).sum(), ref[5]]
            assert np.all(np.abs(m[k, :6] - ref) <= rtol * np.array(scale)), (counts, k, m[k], ref)
    s.close()

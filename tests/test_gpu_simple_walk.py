"""The optics stage for surfaces without rotations, odd or Zernike terms, and the one for all surfaces, against the one-kernel
path of phosim_trace_noalloc, whose walk takes every kind: the same records, images and counts.  A system without those
terms, decentred and shifted, steeply curved (rays that graze or miss a surface take the double-single root), and with
each term in turn; photons and bundles, with and without the dynamic transmission test, kernel by kernel and as a
graph."""
import ctypes as C

import numpy as np
import pytest

from paper_1504_06570_gb300 import phosim as P
from tests import gpu_helpers as G

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


def system(change, counts, bundle):
    sc = G.test_system_scene(sources=G.mixed_sources(counts, seed=5), atmosphere=False)
    sc.sources.bundle = np.asarray(bundle, np.int32)
    sc.sources.bundle_sigma = np.full(len(counts), 0.01)
    mirror, front, back = sc.surfaces[:3]
    mirror.pert, mirror.zern = (0.0,) * 6, ()
    front.pert = back.pert = (0.0,) * 6
    if change == "moved":
        mirror.pert, front.pert, back.pert = (0.1, -0.2, 0.05) + (0.0,) * 3, (0.02, 0.0, 0.0) + (0.0,) * 3, (0.0, 0.0, 0.1) + (0.0,) * 3
    elif change == "steep":                       # the beam is wider than the balls
        front.R, front.kappa, front.alpha, back.R = 14.0, 0.0, (0.0,) * 8, -14.0
    elif change == "rotated":
        front.pert = (0.0, 0.0, 0.0, 1e-4, -2e-4, 3e-4)
    elif change == "zernike":
        mirror.zern = [0.0, 0.0, 0.0, 3e-5, 2e-5]
    elif change == "odd":
        front.alpha = (1e-9, 2e-12, 1e-16, 0, 0, 0, 0, 0)
    return sc


@pytest.mark.parametrize("early, graph", [(False, False), (True, True)])
@pytest.mark.parametrize("change", ["plain", "moved", "steep", "rotated", "zernike", "odd"])
def test_walks_match_one_kernel(change, early, graph):
    counts = [20001, 0, 700, 33]
    s = P.Scene(system(change, counts, [1, 1, 7, 1]), P.MIXED_DS, early_reject=early, graph=graph)
    L = s.L
    L.phosim_trace_noalloc.argtypes = [C.c_void_p, C.POINTER(P.Source), C.c_int, C.POINTER(C.c_uint64),
                                       C.POINTER(C.c_uint64), C.c_void_p, C.c_void_p, C.c_void_p, C.c_void_p]
    out = []
    for one_kernel in (False, True):
        img = torch.zeros((512, 512), dtype=torch.int32, device="cuda")
        rec = torch.zeros(sum(counts) * P.RECORD_DTYPE.itemsize, dtype=torch.uint8, device="cuda")
        if one_kernel:
            rc = L.phosim_trace_noalloc(s.h, s.src, len(counts), s.n_photons.ctypes.data_as(C.POINTER(C.c_uint64)), None,
                                        C.c_void_p(img.data_ptr()), C.c_void_p(rec.data_ptr()), None,
                                        C.c_void_p(torch.cuda.current_stream().cuda_stream))
            assert rc == 0
        else:
            s.trace(img, rec)
            counters = s.counters()
        out.append((img.cpu().numpy(), P.records_to_numpy(rec)))
    s.close()
    (img, rec), (img2, rec2) = out
    assert np.array_equal(rec, rec2) and np.array_equal(img, img2)
    detected = int((rec["flags"] & 1).sum())
    assert int(img.sum()) == detected == int(counters[1])
    fates = np.bincount((rec["flags"] >> 8) & 0xff, minlength=9)
    assert detected > 500 if change != "steep" else fates[2:].sum() > 500

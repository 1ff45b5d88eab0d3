"""The photon counts of a scene's sources as its calls read them: those of the sources, those a program assigns to
Scene.n_photons or writes into the array, in trace as in grad and autotune, and those given to one call.  The library is
replaced by a recorder, so no GPU is needed."""
import ctypes as C
import types

import numpy as np

from paper_1504_06570_gb300 import inputs as I
from paper_1504_06570_gb300 import phosim as P


class Recorder:
    """The library's entry points, which keep the counts that they are given."""

    def __init__(self):
        self.seen = []

    def _keep(self, ptr, n):
        self.seen.append([int(C.cast(ptr, C.POINTER(C.c_uint64))[i]) for i in range(n)])
        return 0

    def phosim_trace(self, h, src, n, counts, *rest):
        return self._keep(counts, n)

    def phosim_grad(self, h, src, n, counts, *rest):
        return self._keep(counts, n)

    def phosim_autotune(self, h, src, n, counts, *rest):
        return self._keep(counts, n)

    def phosim_destroy_scene(self, h):
        return None


def calls(scene):
    scene.L.seen.clear()
    scene.trace(types.SimpleNamespace(data_ptr=lambda: 0), stream=1)
    scene.grad(np.zeros((2, 5)), [(0, 0)], stream=1)
    scene.autotune(stream=1)
    return scene.L.seen


def test_calls_read_the_counts_of_the_moment():
    s = P.Scene.__new__(P.Scene)
    s.L, s.h = Recorder(), 1
    s.set_sources(I.point_sources([0.0, 0.1], [0.0, 0.0], [5, 7]))
    assert calls(s) == [[5, 7]] * 3
    s.n_photons = np.array([11, 0], np.uint64)
    assert calls(s) == [[11, 0]] * 3
    s.n_photons[1] = 13
    assert calls(s) == [[11, 13]] * 3
    s.trace(types.SimpleNamespace(data_ptr=lambda: 0), n_photons=[1, 2], stream=1)
    assert s.L.seen[-1] == [1, 2] and calls(s) == [[11, 13]] * 3
    s.set_sources(I.point_sources([0.0, 0.1], [0.0, 0.0], [3, 4]))
    assert calls(s) == [[3, 4]] * 3

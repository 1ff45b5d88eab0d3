"""Calls on a device with little room left: the adjoint's kept states give way to the photon batches, to scratch that the
scene needs later, and batches and ghosts' buffers are made for smaller chunks of photons.  Images and counts are those of
the same call with room; gradients agree to the order of their sums (1e-9 of a parameter's largest, as in
test_gpu_grad_tape)."""
import numpy as np
import pytest

from paper_1504_06570_gb300 import inputs as I
from paper_1504_06570_gb300 import phosim as P
from tests import gpu_helpers as G
from tests.test_gpu_ghost_rounds import ghost_scene

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]

PARAMS = [(1, 0), (2, 1), (5, 2)]


class Room:
    """Holds all of the device's free memory but so many MB."""

    def __init__(self, megabytes):
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        self.hold = torch.empty(torch.cuda.mem_get_info()[0] - (megabytes << 20), dtype=torch.uint8, device="cuda")

    def __enter__(self):
        return self

    def __exit__(self, *_):
        torch.cuda.synchronize()
        del self.hold
        torch.cuda.empty_cache()


def field(photons, pass_part):
    sc = G.test_system_scene(sources=G.mixed_sources([photons, photons // 3], seed=6), atmosphere=False)
    sc.coatings = [I.Coating(lam0=400.0, dlam=300.0, theta0=0.0, dtheta=1.6, table=np.array([[pass_part]]))]
    return sc


def image(sc):
    return torch.zeros((sc.detector.ny, sc.detector.nx), dtype=torch.int32, device="cuda")


def warmed(sc, precision, call=lambda s, few: None):
    """A scene whose kernels are loaded by a small call of the same kinds."""
    s = P.Scene(sc, precision, early_reject=precision != P.MIXED_DS)
    few = np.full(len(sc.sources), 500, np.uint64)
    s.trace(image(sc), n_photons=few)
    call(s, few)
    return s


# batches of 8e7 photons: 360 MB; kept states of a system of six surfaces: 512 MB and one a warp (43 MB); so of 750 MB both do
# not fit, of 250 MB the batches of half of the photons do
@pytest.mark.parametrize("megabytes", [750, 250])
def test_gradient(megabytes):
    sc, dL = field(60_000_000, 0.02), np.random.default_rng(2).normal(size=(2, 5))
    s = P.Scene(sc, P.PLAIN_FP64)
    g, m = s.grad(dL, PARAMS)
    s.close()
    s = warmed(sc, P.PLAIN_FP64, lambda s, few: s.grad(dL, PARAMS, n_photons=few))
    with Room(megabytes):
        for _ in range(2):
            g2, m2 = s.grad(dL, PARAMS)
            assert np.array_equal(m[:, 0], m2[:, 0]) and m[0, 0] > 1000
            assert np.all(np.abs(g2 - g) <= 1e-9 * np.abs(g).max(axis=0))
    s.close()


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("precision", [P.PLAIN_FP64, P.MIXED])
def test_batches_in_smaller_chunks(precision, graph):
    sc = field(60_000_000, 0.02)
    ref = G.run_gpu(sc, precision, records=False, moments=False, early_reject=True, graph=graph)
    s = warmed(sc, precision)
    img = image(sc)
    with Room(200):
        s.trace(img)
        counters = s.counters()
        assert np.array_equal(img.cpu().numpy().view(np.uint32), ref["image"])
        assert np.array_equal(counters, ref["counters"])
    s.close()


def test_ghosts_in_smaller_chunks():
    # 261 bytes a photon: 3.1 GB
    sc = ghost_scene([7_000_000, 5_000_000], 0.3, 1)
    ref = G.run_gpu(sc, P.MIXED_DS, records=False, moments=False)
    s = warmed(sc, P.MIXED_DS)
    img = image(sc)
    with Room(1200):
        s.trace(img)
        counters = s.counters()
        assert np.array_equal(img.cpu().numpy().view(np.uint32), ref["image"])
        assert np.array_equal(counters, ref["counters"])
    s.close()


def test_batches_take_the_kept_states():
    # a gradient of 3e6 photons keeps 512 MB of states; a trace of 8e7 wants 360 MB of batches, and there are 60
    sc, dL = field(60_000_000, 0.02), np.ones((2, 5))
    ref = G.run_gpu(sc, P.PLAIN_FP64, records=False, moments=False, early_reject=True)
    some = np.array([2_000_000, 1_000_000], np.uint64)
    s = warmed(sc, P.PLAIN_FP64, lambda s, few: s.grad(dL, PARAMS, n_photons=few))
    g, _ = s.grad(dL, PARAMS, n_photons=some)
    img = image(sc)
    with Room(60):
        s.trace(img)
        assert np.array_equal(img.cpu().numpy().view(np.uint32), ref["image"])
        again, _ = s.grad(dL, PARAMS, n_photons=some)
    for other in (again, s.grad(dL, PARAMS, n_photons=some)[0]):
        assert np.all(np.abs(other - g) <= 1e-9 * np.abs(g).max(axis=0))
    s.close()

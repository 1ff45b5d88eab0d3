"""The adjoint's forward states: kept by the forward pass (with a coated surface, whose dynamic transmission test makes
batches of the photons that go on, up to 512 MB of them) or traced again.  A scene whose coating passes everything against
the same without coatings; the sweep ending at a later surface; and a source alone against the same source in a list with
more photons than the states kept, whichever of its batches those then are.  The sums differ in their order only: 1e-9 of a
parameter's largest gradient, for up to 3e4 additions in FP64 whose terms cancel to a thousandth at most."""
import numpy as np
import pytest

from paper_1504_06570_gb300 import inputs as I
from paper_1504_06570_gb300 import phosim as P
from tests import gpu_helpers as G

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]

PARAMS = [(0, 3), (0, 104), (1, 0), (2, 1), (3, 4), (5, 0), (5, 2)]


def gradient(sc, params, dL, repeat=1):
    s = P.Scene(sc, P.PLAIN_FP64)
    for _ in range(repeat):
        g, m = s.grad(dL, params)
    s.close()
    return g, m


def close(a, b):
    return np.all(np.abs(a - b) <= 1e-9 * np.abs(b).max(axis=0))


@pytest.mark.parametrize("counts, bundle", [([1], 1), ([31, 0, 33], 1), ([5000, 64, 777], 1), ([4000, 30], 6)])
@pytest.mark.parametrize("first", [0, 3])
def test_kept_states_are_those_traced_again(counts, bundle, first):
    sc = G.test_system_scene(sources=G.mixed_sources(counts, seed=6), atmosphere=False)
    sc.sources.bundle = np.full(len(counts), bundle, np.int32)
    sc.sources.bundle_sigma = np.full(len(counts), 0.01)
    params = [p for p in PARAMS if p[0] >= first]
    dL = np.random.default_rng(2).normal(size=(len(counts), 5))
    sc.coatings = [I.Coating(lam0=400.0, dlam=300.0, theta0=0.0, dtheta=1.6, table=np.array([[1.0]]))]
    g, m = gradient(sc, params, dL, repeat=2)
    sc.surfaces[3].coating = -1
    g2, m2 = gradient(sc, params, dL)
    assert np.array_equal(m[:, 0], m2[:, 0]) and m[0, 0] > 0
    assert close(g, g2), (g, g2)


def test_more_photons_than_states_kept():
    counts = [100000, 4000000]
    sc = G.test_system_scene(sources=G.mixed_sources(counts, seed=6), atmosphere=False)
    sc.coatings = [I.Coating(lam0=400.0, dlam=300.0, theta0=0.0, dtheta=1.6, table=np.array([[0.9]]))]
    dL = np.random.default_rng(3).normal(size=(2, 5))
    both, _ = gradient(sc, PARAMS, dL)
    sc.sources = G.mixed_sources(counts[:1], seed=6)
    reference = G.test_system_scene(sources=G.mixed_sources(counts, seed=6), atmosphere=False).sources
    for name in ("xi", "eta", "t0", "pa"):
        getattr(sc.sources, name)[:] = getattr(reference, name)[:1]
    alone, _ = gradient(sc, PARAMS, dL[:1])
    assert close(both[:1], alone), (both[0], alone[0])

"""The adjoint of a surface as a rigid body (force and torque) and of its figure's second derivatives, against the oracle's
forward-mode dual numbers: each surface in turn, mirror, lens, plate and detector, all of them shifted and turned about
every axis and the mirror with all 28 Zernike terms, with and without the sensor.  Both are exact derivatives in FP64 in
another order, so the tolerance is that of the repository's other comparison of the two, 1e-6 of a parameter's largest
gradient."""
import numpy as np
import pytest

from paper_1504_06570_gb300 import phosim as P
from tests import gpu_helpers as G
from tests.test_gpu_grad import oracle_gradient

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


@pytest.mark.parametrize("sensor", [True, False])
@pytest.mark.parametrize("surface", range(6))
def test_rigid_body_matches_oracle(oracle_mod, surface, sensor):
    counts = [2000, 600, 31]
    sc = G.test_system_scene(sources=G.mixed_sources(counts, seed=9), atmosphere=False, sensor=sensor)
    rng = np.random.default_rng(17)
    for k, s in enumerate(sc.surfaces):
        turn = 2e-6 if k == 0 else 2e-3
        s.pert = tuple(rng.normal(size=3) * 0.02) + tuple(rng.normal(size=3) * turn)
    sc.surfaces[0].zern = list(rng.normal(size=28) * 1e-5)
    params = [(surface, f) for f in range(6)] + [(0, 104), (0, 127)]
    dL = rng.normal(size=(len(counts), 5))
    s = P.Scene(sc, P.PLAIN_FP64)
    g, _ = s.grad(dL, params)
    s.close()
    go = oracle_gradient(oracle_mod, sc, dL, params)
    scale = np.abs(go).max(axis=0) + 1e-300
    assert np.all(np.abs(g - go) <= 1e-6 * scale), ((np.abs(g - go) / scale).max(axis=0), g[0], go[0])

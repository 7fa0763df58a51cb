"""Initial frames of rods folded back on themselves: the directors after the fold are still unit
vectors normal to their tangents, as those of a chain that normalises at every edge are.

The scan works in FP64 on unit turns, so what is left is the rounding of the components to float32
(6e-8 each at most): 1.3e-7 in the length and, with the tangent's own, 2.6e-7 across it."""
import numpy as np
import pytest
import torch

from paper_2606_04206_gb300 import inputs
from gpu_util import sim_for

pytestmark = pytest.mark.gpu

FOLDS = (1e-1, 1e-3, 1e-4, 1e-5, 3e-6, 1e-6, 3e-7)


def folded(rng, n, delta):
    """Unit steps along a random direction, back at pi - delta, then along two others."""
    R = np.linalg.qr(rng.normal(size=(3, 3)))[0]
    m = n // 3
    d = np.concatenate([np.tile([1.0, 0.0, 0.0], (m, 1)), [[-np.cos(delta), np.sin(delta), 0.0]],
                        np.tile([0.3, 0.8, 0.2], (m, 1)), np.tile([0.1, 0.7, -0.4], (n - 2 - 2 * m, 1))])
    x = np.concatenate([np.zeros((1, 3)), np.cumsum(d * 0.01, 0)])
    return (x - x[m]) @ R.T   # the fold at the origin, where float32 resolves it


@pytest.mark.parametrize("n", [5, 40, 200])
def test_directors_stay_unit_vectors(n):
    rng = np.random.default_rng(n)
    line = np.stack([0.01 * np.arange(n), np.zeros(n), np.full(n, 0.5)], 1)
    p = inputs.custom([line] * len(FOLDS), K=1e5, E=1e4, G=1e3)
    sim = sim_for(p)
    x, v, th = sim.tensors_from_problem()
    x[:, :3] = torch.as_tensor(np.concatenate([folded(rng, n, d) for d in FOLDS]), dtype=torch.float32)
    sim.set_state(x, v, th)
    ref, tan, hinge, _ = (a.double().cpu().numpy() for a in sim.get_internal())
    length = np.linalg.norm(ref[:, :3], axis=1).reshape(len(FOLDS), n - 1)
    across = np.abs((ref[:, :3] * tan[:, :3]).sum(1)).reshape(len(FOLDS), n - 1)
    assert np.abs(length - 1.0).max() <= 1.3e-7, np.abs(length - 1.0).max(1)
    assert across.max() <= 2.6e-7, across.max(1)
    assert not hinge[:, 3].any()

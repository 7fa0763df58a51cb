"""The self-repulsion penalty at distances on both sides of nine tenths of the rod's reach (the
farthest vertex from the first), where the kernel stops testing spheres, and far beyond; against the
FP64 definition with the bars of test_gpu_losses.py."""
import numpy as np
import pytest
import torch

from oracle import losses as L
from paper_2606_04206_gb300 import dlo, inputs
from gpu_util import sim_for
from test_gpu_losses import check, per_rod

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("closed", [False, True])
@pytest.mark.parametrize("reach", [0.2, 0.89, 0.91, 1.5, 10.0])
def test_reach(reach, closed):
    sizes = (4, 9, 33, 128, 256)
    rng = np.random.default_rng(len(sizes))
    rods = []
    for n in sizes:
        s = np.linspace(0.0, 2 * np.pi if closed else 1.8 * np.pi, n, endpoint=not closed)
        x = np.stack([np.sin(s) + 2 * np.sin(2 * s), np.cos(s) - 2 * np.cos(2 * s), -np.sin(3 * s)], 1)
        rods.append(0.06 * x + rng.normal(size=(n, 3)) * 0.06 / n + [0.0, 0.0, 0.3])
    p = inputs.custom(rods, closed=[closed] * len(rods), K=1e5, E=1e4)
    sim = sim_for(p)
    x = sim.tensors_from_problem()[0]
    g = torch.as_tensor(rng.uniform(0.5, 2.0, p.batch), dtype=torch.float32, device="cuda")
    far = [max(np.linalg.norm(r - r[0], axis=1)) for r in rods]
    prm = torch.tensor([[reach * f, 1.0, 0.0, 0.0] for f in far], dtype=torch.float32, device="cuda")
    q, gx = sim.loss(dlo.LOSS_REPULSION, x, prm, g)
    delta = prm[:, 0].double().cpu()
    q_ref, g_ref = per_rod(p, x, lambda b, xb: L.repulsion(xb, float(delta[b]), 1, closed=closed) + 0.0 * xb.sum())
    for b in range(p.batch):   # each rod by its own size: the penalties grow with the square of the distance
        assert abs(float(q[b]) - q_ref[b]) <= 1e-4 * (1.0 + abs(q_ref[b]))
    check(q, gx, q_ref, g_ref, g, p, 1e-4)

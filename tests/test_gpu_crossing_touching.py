"""The crossing loss of rods with two vertices of non-adjacent edges at (or nearly at) one point:
a ring given as an open rod whose last vertex repeats its first, and a rod that touches itself.

A pair's angle is the sum of two arctangents.  The triple product of either comes from vectors at
most four times as long as the shortest that enters its denominator, or is formed of the
triangle's own vectors, so it is off by at most some 16 roundings (16 x 6e-8) of the
denominator and the angle by 1e-6; over the few pairs at the shared point and 1 / (4 pi) each, and
with the roundings of the others (below 2e-6 at these sizes), 1e-5 (1 + |Q|) holds with a margin."""
import numpy as np
import pytest
import torch

from oracle import losses as L
from paper_2606_04206_gb300 import dlo, inputs
from gpu_util import grad_agreement, sim_for

pytestmark = pytest.mark.gpu


def ring(n, gap):
    s = np.linspace(0.0, 2 * np.pi, n)
    x = 0.06 * np.stack([np.sin(s) + 2 * np.sin(2 * s), np.cos(s) - 2 * np.cos(2 * s), -np.sin(3 * s)], 1)
    x[-1] = x[0] + gap * np.array([0.3, 0.5, 0.8])
    return x


def touching(n, gap):
    x = ring(n, 0.01)
    x[2 * n // 3] = x[n // 5] + gap * np.array([0.3, -0.5, 0.8])
    return x


@pytest.mark.parametrize("shape", [ring, touching])
@pytest.mark.parametrize("sizes", [(8, 33, 40, 128), (20, 129, 256)])
@pytest.mark.parametrize("gap", [0.0, 1e-8, 1e-6, 1e-5, 1e-3])
def test_value_and_gradient(shape, sizes, gap):
    p = inputs.custom([ring(n, 0.01) + [0.0, 0.0, 0.3] for n in sizes], K=1e5, E=1e4)   # rest shape
    sim = sim_for(p)
    x = torch.zeros(sim.V, 4, device="cuda")
    x[:, :3] = torch.as_tensor(np.concatenate([shape(n, gap) for n in sizes]), dtype=torch.float32)
    q_only, _ = sim.loss(dlo.LOSS_CROSSING, x, grad=False)
    q, gx = sim.loss(dlo.LOSS_CROSSING, x)
    xs = x[:, :3].double().cpu()
    for b in range(p.batch):
        v = slice(p.vert_off[b], p.vert_off[b + 1])
        xb = xs[v].clone().requires_grad_(True)
        ref = L.crossing(xb)
        tol = 1e-5 * (1.0 + abs(float(ref.detach())))
        assert abs(float(q_only[b]) - float(ref.detach())) <= tol, (b, float(q_only[b]), float(ref.detach()))
        assert abs(float(q[b]) - float(ref.detach())) <= tol, (b, float(q[b]), float(ref.detach()))
        # at the point itself the angle has no gradient; above 128 vertices the gradient comes from
        # dual numbers, which near a shared point are only good to some 1e-3 of it
        if gap >= 1e-5 and max(sizes) <= 128:
            rel, cos = grad_agreement(gx[v, :3].double().cpu().numpy(), torch.autograd.grad(ref, [xb])[0].numpy())
            assert rel <= 1e-3 and cos >= 0.999, (b, rel, cos)

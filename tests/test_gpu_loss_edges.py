"""The crossing, repulsion and silhouette losses at the sizes where their kernels change shape:
the smallest rods, one edge more or less than a warp and than a CTA, the largest; images that
are not whole tiles.  Against the FP64 definitions, with the bars of test_gpu_losses.py and
test_gpu_silhouette.py."""
import math

import numpy as np
import pytest
import torch

from oracle import losses as L
from oracle.silhouette import camera, render, silhouette_loss
from paper_2606_04206_gb300 import dlo, inputs
from gpu_util import grad_agreement, sim_for
from test_gpu_losses import check, per_rod

pytestmark = pytest.mark.gpu


def tangle(rng, n, closed):
    """A space curve that passes over itself several times, with a little roughness."""
    s = np.linspace(0.0, 2 * np.pi, n, endpoint=not closed)
    f = s if closed else 0.9 * s
    x = np.stack([np.sin(f) + 2 * np.sin(2 * f), np.cos(f) - 2 * np.cos(2 * f), -np.sin(3 * f)], 1)
    return 0.06 * x + rng.normal(size=(n, 3)) * 0.06 / n + [0.0, 0.0, 0.3]


def case(sizes, closed):
    rng = np.random.default_rng(sum(sizes))
    rods = [tangle(rng, n, closed) for n in sizes]
    p = inputs.custom(rods, closed=[closed] * len(rods), K=1e5, E=1e4)
    sim = sim_for(p)
    x = sim.tensors_from_problem()[0]
    g = torch.as_tensor(rng.uniform(0.5, 2.0, p.batch), dtype=torch.float32, device=x.device)
    return p, sim, x, g


SIZES = [(False, (4, 5, 32, 33, 34, 128)), (False, (127, 129, 193, 256)), (True, (4, 5, 32, 33, 65, 128)), (True, (64, 200, 255))]


@pytest.mark.parametrize("closed,sizes", SIZES)
def test_crossing_and_repulsion_at_every_size(closed, sizes):
    p, sim, x, g = case(sizes, closed)
    q, gx = sim.loss(dlo.LOSS_CROSSING, x, None, g)
    q_ref, g_ref = per_rod(p, x, lambda b, xb: L.crossing(xb, closed=closed) + 0.0 * xb.sum())
    check(q, gx, q_ref, g_ref, g, p, 2e-4)
    q_only, none = sim.loss(dlo.LOSS_CROSSING, x, None, g, grad=False)   # each pair once, not twice
    assert none is None and float((q_only - q).abs().max()) <= 2e-4 * (1.0 + float(q.abs().max()))
    prm = torch.tensor([[0.05, 2.0, 0.0, 0.0]] * p.batch, device=x.device)
    q, gx = sim.loss(dlo.LOSS_REPULSION, x, prm, g)
    q_ref, g_ref = per_rod(p, x, lambda b, xb: L.repulsion(xb, float(np.float32(0.05)), 2, closed=closed) + 0.0 * xb.sum())
    check(q, gx, q_ref, g_ref, g, p, 1e-4)


@pytest.mark.parametrize("height,width", [(5, 3), (8, 32), (9, 33), (7, 70), (50, 31)])
@pytest.mark.parametrize("closed", [False, True])
def test_silhouette_at_odd_image_sizes(height, width, closed):
    p, sim, x, g = case((3, 40, 130), closed)
    rng = np.random.default_rng(height * width)
    f, tau = 0.9 * max(height, width), 0.6
    a = math.radians(50.0)
    R = np.array([[1.0, 0.0, 0.0], [0.0, -math.sin(a), -math.cos(a)], [0.0, math.cos(a), -math.sin(a)]])
    eye = np.array([0.0, -math.cos(a), math.sin(a)]) * 0.9
    cams = np.stack([camera(f, f, width / 2, height / 2, np.diag([1.0, -1.0, -1.0]), [0.0, 0.0, 1.2]),
                     camera(f, f, width / 2, height / 2, R, -R @ eye)])
    masks = (rng.uniform(size=(p.batch, 2, height, width)) < 0.3).astype(np.uint8)
    q, gx, img = sim.silhouette(x, torch.tensor(cams, dtype=torch.float32, device="cuda"), torch.tensor(masks, device="cuda"),
                                tau, g, render=True)
    q_only, none, _ = sim.silhouette(x, torch.tensor(cams, dtype=torch.float32, device="cuda"),
                                     torch.tensor(masks, device="cuda"), tau, g, grad=False)
    assert none is None and torch.equal(q_only, q)
    xs = x[:, :3].double().cpu()
    for b in range(p.batch):
        v0, v1 = p.vert_off[b], p.vert_off[b + 1]
        xb = xs[v0:v1].clone().requires_grad_(True)
        r = float(p.radius[b])
        loss = silhouette_loss(xb, cams, masks[b], tau, r, closed)
        gb, = torch.autograd.grad(loss, [xb])
        loss = float(loss.detach())
        assert abs(float(q[b]) - loss) <= 1e-4 * loss + 1e-7
        rel, cos = grad_agreement(gx[v0:v1, :3].double().cpu().numpy(), float(g[b]) * gb.numpy())
        assert rel <= 1e-3 and cos >= 0.999, (b, rel, cos)
        for c in range(2):
            o = render(xb.detach(), cams[c], height, width, tau, r, closed)
            assert np.abs(img[b, c].double().cpu().numpy() - o.numpy()).max() <= 2e-5

"""The fused step and its adjoint at the edges of the kernels' warps, size classes and projection
buffers, against the FP64 oracle: elastic, inextensible and strain-limited rods side by side,
open and closed (odd loops have a third projection colour), from a bent start above the table.

Bars: those of tests/test_gpu_forward.py (positions to 1e-5 of their size, velocities to 2e-3,
twist angles to 1e-4 after a frame) and of tests/test_gpu_backward.py (relative L2 1e-3), for
velocities and gradients or twice what the oracle's own definitions miss in float32 where that is
more: on a rod of 2 m float32 positions resolve the strain of its 8 mm edges to 1.5e-5 only."""
import numpy as np
import pytest
import torch

from oracle import OracleSim
from paper_2606_04206_gb300 import inputs
from gpu_util import actions_dev, device_gradients, grad_agreement, oracle_gradients, rel_inf, sim_for
from test_gpu_backward import GROUPS, log_sens, weights

pytestmark = pytest.mark.gpu


def rods(n, closed, frames=1, **kw):
    """Three rods of n vertices 8 mm apart: a bent curve in space, not near itself."""
    rng = np.random.default_rng([n, closed])
    out = []
    for _ in range(3):
        L = 0.008 * n
        s = np.linspace(0, 2 * np.pi, n, endpoint=not closed)
        r = L / (2 * np.pi)
        x = np.stack([r * np.cos(s), r * np.sin(s), 0.1 * r * np.sin(2 * s)], 1) if closed else \
            np.stack([L * s / (2 * np.pi), 0.1 * L * np.sin(s + rng.uniform(0, 6)), 0.05 * L * np.cos(s)], 1)
        out.append(x + [0, 0, 0.2 + 0.3 * r] + rng.normal(0, 1e-4, (n, 3)))
    kind = np.arange(3)
    p = inputs.custom(out, closed=[closed] * 3, frames=frames, K=np.where(kind == 1, 0.0, 1e5), E=1e4,
                      G=np.where(kind == 0, 0.0, 1e3), inextensible=kind == 1, strain_limit=np.where(kind == 2, 2e-4, 0.0),
                      planes=np.array([[0.0, 0.0, 1.0, 0.0]]), self_contact=True, **kw)
    t = np.linspace(0, 2 * np.pi, n)[:, None]
    p.v0 = inputs.f32(np.tile(0.1 * np.sin(2 * t + [0.3, 1.1, 2.0]), (3, 1)))   # stretches edges past the strain limit
    return p


OPEN = [2, 3, 4, 31, 32, 33, 63, 64, 65, 127, 128, 129, 192, 193, 224, 225, 256]
CLOSED = [5, 31, 32, 33, 63, 64, 65, 127, 128, 129, 191, 192, 193, 223, 224, 225, 255, 256]


def frame_of_oracle(p, dtype):
    o = OracleSim(p, dtype=dtype)
    o.set_state(p.x0, p.v0, p.theta0, p.omega0)
    o.step(p.actions, 1)
    return o.get_state()


@pytest.mark.parametrize("n,closed", [(n, False) for n in OPEN] + [(n, True) for n in CLOSED])
def test_one_frame(n, closed):
    p = rods(n, closed)
    sim = sim_for(p)
    sim.reset()
    sim.step(actions_dev(p), 1)
    a, b, c = sim.full_state_numpy(), frame_of_oracle(p, torch.float64), frame_of_oracle(p, torch.float32)
    floor = rel_inf(c["v"], b["v"])
    assert rel_inf(a["x"], b["x"]) <= 1e-5
    assert rel_inf(a["v"], b["v"]) <= max(2e-3, 2 * floor)
    assert np.abs(a["theta"] - b["theta"]).max() <= 1e-4
    assert not sim.query(2).any()


@pytest.mark.parametrize("n,closed,n_iter", [(33, True, 11), (64, True, 11), (65, False, 23), (128, False, 1),
                                             (127, True, 10), (129, True, 5), (200, False, 13), (256, True, 6), (255, True, 4)])
def test_gradient_of_a_frame(n, closed, n_iter):
    """n_iter on both sides of the iterations whose records are fetched ahead (5 or 10 by class)."""
    p = rods(n, closed)
    p.n_iter = n_iter
    wx, wv, wth = weights(p, 0)
    ref, _ = oracle_gradients(p, 1, wx, wv, wth)
    f32, _ = oracle_gradients(p, 1, wx, wv, wth, dtype=torch.float32)
    got = device_gradients(sim_for(p), p, 1, wx, wv, wth)
    for g in (got, ref, f32):
        g["material"] = log_sens(p, g["material"])
    for k in GROUPS:
        rel, _ = grad_agreement(got[k], ref[k])
        floor, _ = grad_agreement(f32[k], ref[k])
        assert rel <= max(1e-3, 2 * floor), (k, rel, floor)

"""The three kernels that step a rod (forward, forward with records, recompute) round alike: hinges
on their yield surface branch on the last bit of their curvature.  Figure-eight rods and loops of
every size class that yield all along and, with self-contact, touch at their crossing: the state of a
recorded step equals that of an unrecorded one bit for bit (contact corrections are summed in fixed
point, so their order does not matter), and the gradient on stored records equals the recomputed one,
bit for bit without contact and to 1e-4 of each rod's with it (float atomics; a hinge that yields in
one and not in the other changes its rod's by more than 1e-3)."""
import numpy as np
import pytest
import torch

from paper_2606_04206_gb300 import inputs
from paper_2606_04206_gb300.dlo import Q_LAUNCHES, Q_PAIRS
from gpu_util import actions_dev, sim_for
from test_gpu_backward import weights

pytestmark = pytest.mark.gpu

LOW = {32: 17, 64: 33, 128: 65, 192: 129, 224: 193, 256: 225}


def eights(n, contact):
    """Per class: sizes over its range, open and closed, elastic with and without torsion, cables,
    strain-limited, all plastic."""
    rng = np.random.default_rng(n)
    rods, closed, kind = [], [], []
    r = 0.002
    for b in range(40):
        nv, loop = int(rng.integers(LOW[n], n + 1)), b % 3 == 2
        s = np.linspace(0.0, 2 * np.pi, nv, endpoint=not loop) * (1.0 if loop else 0.97)
        size = 0.008 * nv / 4.0
        lift = r * (1.02 if contact else 3.0)
        x = np.stack([0.6 * size * np.sin(2 * s), size * np.sin(s), lift * np.cos(s)], 1)
        rods.append(x + [0.0, 0.0, 0.3] + rng.normal(size=(nv, 3)) * 2e-5)
        closed.append(loop)
        kind.append(b % 4)
    kind = np.array(kind)
    p = inputs.custom(rods, closed=closed, frames=2, E=1e5, K=np.where(kind == 2, 0.0, 1e5),
                      G=np.where(kind == 1, 0.0, 4e4), inextensible=kind == 2, strain_limit=np.where(kind == 3, 0.02, 0.0),
                      plastic=np.ones(40, bool), yield_curv=np.full(40, 0.5), self_contact=contact)
    p.v0[:] = inputs.f32(rng.normal(size=p.v0.shape) * 0.2)
    p.omega0[:] = inputs.f32(rng.normal(size=p.omega0.shape) * 5.0)
    return p


@pytest.mark.parametrize("contact", [False, True])
@pytest.mark.parametrize("n", sorted(LOW))
def test_recorded_unrecorded_and_recomputed_agree(n, contact):
    p = eights(n, contact)
    sim = sim_for(p)
    w = [torch.as_tensor(a, dtype=torch.float32, device="cuda") for a in weights(p, 2)]
    states, grads, launches = [], [], []
    for run in range(3):   # unrecorded; recorded, recomputed; recorded, stored
        sim.reset()
        if run:
            sim.begin_rollout(2)
        sim.step(actions_dev(p), 2)
        states.append(sim.full_state_numpy())
        if run:
            before = sim.query(Q_LAUNCHES)
            grads.append(sim.backward(*w))
            launches.append(sim.query(Q_LAUNCHES) - before)
    assert launches == [3, 2]   # recompute, reverse, frames; reverse, frames
    if contact:
        assert (sim.query(Q_PAIRS) > 0).sum() >= 30
    assert np.abs(states[0]["kbar"]).max() > 0.0
    for k in states[0]:
        assert np.array_equal(states[0][k], states[1][k]) and np.array_equal(states[0][k], states[2][k]), k
    vo, eo = p.vert_off, p.edge_off
    for k in grads[0]:
        a, b = (g[k].double().cpu().numpy() for g in grads)
        assert np.isfinite(a).all(), k
        if not contact:
            assert np.array_equal(a, b), k
            continue
        for rod in range(p.batch):
            sl = {"actions": (slice(None), rod), "material": rod, "x0": slice(vo[rod], vo[rod + 1]),
                  "v0": slice(vo[rod], vo[rod + 1]), "theta0": slice(eo[rod], eo[rod + 1])}[k]
            assert np.linalg.norm(a[sl] - b[sl]) <= 1e-4 * np.linalg.norm(a[sl]), (k, rod)

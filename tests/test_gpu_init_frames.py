"""The initial reference frames (dlo_set_state) as a scan over a rod's edges, against the chain of
space-parallel transports it replaces, walked edge by edge in FP64, and its adjoint against the
FP64 oracle, at the edges of the scan's warps and of the size classes.

Both sides are FP64 up to the final rounding to float32, so a unit director's components agree
within one rounding of a number below 1 (6e-8) plus the chain's own FP64 error (256 x 2e-16)."""
import numpy as np
import pytest
import torch

from paper_2606_04206_gb300 import inputs
from gpu_util import device_gradients, grad_agreement, oracle_gradients, sim_for
from test_gpu_backward import weights

pytestmark = pytest.mark.gpu


def curve(rng, n, closed):
    s = np.linspace(0, 2 * np.pi, n, endpoint=not closed)
    x = np.stack([np.cos(s) if closed else 0.8 * s, np.sin(s) + 0.2 * np.sin(2 * s), 0.3 * np.sin(3 * s + 1)], 1)
    return 0.2 * x + rng.uniform(-0.1, 0.1, 3) + [0, 0, 1]


def chain(x, closed, starts):
    """(d1, reference twist at each vertex) by walking the rod."""
    unit = lambda a: a / np.linalg.norm(a)
    n, ne = len(x), len(x) - 1 + closed
    t = [unit(x[(j + 1) % n] - x[j]) for j in range(ne)]
    brk = [not closed and (j + 1) in starts for j in range(ne)]
    adapt = lambda d, t: unit(d - (d @ t) * t)
    first = lambda t: adapt(np.array([0.0, 0, 1] if abs(t[2]) < 0.9 else [1.0, 0, 0]), t)

    def move(a, b, d):
        k = np.cross(a, b)
        return (a @ b) * d + np.cross(k, d) + (k @ d) / (1 + a @ b) * k

    d = []
    for j in range(ne):
        if brk[j]:
            t[j] = np.array([0.0, 0, 1])
            d.append(np.array([1.0, 0, 0]))
        else:
            d.append(first(t[j]) if j == 0 or brk[j - 1] else adapt(move(t[j - 1], t[j], d[-1]), t[j]))
    if closed:
        u = adapt(move(t[-1], t[0], d[-1]), t[0])
        psi = np.arctan2(np.cross(d[0], u) @ t[0], d[0] @ u)
        for j in range(ne):
            p = -psi * j / ne
            d[j] = np.cos(p) * d[j] + np.sin(p) * np.cross(t[j], d[j])
    m = np.zeros(n)
    for b in range(0 if closed else 1, ne):
        a = b - 1 if b else ne - 1
        if not (brk[a] or brk[b]):
            u = move(t[a], t[b], d[a])
            m[b] = np.arctan2(np.cross(u, d[b]) @ t[b], u @ d[b])
    return np.array(d), m


@pytest.mark.parametrize("closed,sizes", [(False, (2, 3, 32, 33, 34, 64, 65, 66, 129, 193, 256)), (True, (3, 32, 33, 64, 65, 128, 225, 256))])
def test_frames_match_the_chain(closed, sizes):
    rng = np.random.default_rng(len(sizes))
    rods = [curve(rng, n, closed) for n in sizes]
    p = inputs.custom(rods, closed=[closed] * len(rods), K=1e5, E=1e4, G=1e3)
    check_frames(p, [()] * len(rods))


def test_frames_of_strands_start_afresh():
    rng = np.random.default_rng(3)
    starts = [(5,), (31, 33), (64,), (2, 250)]
    rods = [np.concatenate([curve(rng, b - a, False) + 0.3 * a for a, b in zip((0,) + s, s + (n,))])
            for s, n in zip(starts, (12, 70, 66, 256))]
    p = inputs.custom(rods, K=0.0, E=1e4, G=1e3, inextensible=True)
    for b, s in enumerate(starts):
        p.strand_start[p.vert_off[b] + np.array(s)] = True
    check_frames(p, starts)


def check_frames(p, starts):
    sim = sim_for(p)
    sim.reset()
    ref, tan, hinge, _ = (a.double().cpu().numpy() for a in sim.get_internal())
    for b in range(p.batch):
        v, e = slice(p.vert_off[b], p.vert_off[b + 1]), slice(p.edge_off[b], p.edge_off[b + 1])
        d, m = chain(p.x0[v], bool(p.closed[b]), starts[b])
        assert np.abs(ref[e, :3] - d).max() <= 1.3e-7, (b, np.abs(ref[e, :3] - d).max())
        assert np.abs(hinge[v, 3] - m).max() <= 1.3e-7 * np.pi, (b, np.abs(hinge[v, 3] - m).max())
        assert np.array_equal(hinge[v, 2], hinge[v, 3])   # x0 is the rest shape: rest twist = reference twist


@pytest.mark.parametrize("closed,n", [(False, 2), (False, 3), (False, 33), (False, 65), (True, 3), (True, 33), (True, 64)])
def test_frames_adjoint_matches_the_oracle(closed, n):
    """dL/dx0 through the frames, for twisted rods whose frames matter; the bar of the other
    gradient tests (1e-3, cosine 0.999)."""
    rng = np.random.default_rng(n)
    p = inputs.custom([curve(rng, n, closed) for _ in range(2)], closed=[closed] * 2, frames=2, K=1e5, E=1e5, G=1e5)
    p.theta0[:] = inputs.f32(rng.uniform(-0.5, 0.5, len(p.theta0)))
    w = weights(p, 1)
    ref, _ = oracle_gradients(p, 2, *w)
    got = device_gradients(sim_for(p), p, 2, *w)
    for k in ("x0", "v0", "th0"):
        rel, cos = grad_agreement(got[k], ref[k])
        assert rel <= 1e-3 and cos >= 0.999, (k, rel, cos)

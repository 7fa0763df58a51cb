"""The backward on the substep records the forward stored, against the backward that steps again
to get them (a budget too small for the records of the whole rollout): the same values bit for
bit where no candidates are involved, and to float accumulation order where they are."""
import numpy as np
import pytest
import torch

from paper_2606_04206_gb300 import inputs
from gpu_util import actions_dev, sim_for
from test_gpu_backward import weights

pytestmark = pytest.mark.gpu


def gradients(p, frames, chunks=None, substeps=0, plain_first=False, **opt):
    sim = sim_for(p, **opt)
    wx, wv, wth = (torch.as_tensor(w, dtype=torch.float32, device="cuda") for w in weights(p, 2))
    sim.reset()
    sim.begin_rollout(frames)
    f = 0
    for n in chunks or (frames,):
        sim.step(actions_dev(p, f, f + n), n, substeps)
        f += n
    before = sim.query(7)
    if plain_first:   # takes over the workspace the records are in
        sim.backward(wx, wv, wth, plain=True)
    out = [sim.backward(wx, wv, wth) for _ in range(2)]
    assert all(torch.equal(out[0][k], out[1][k]) for k in out[0]) or p.self_contact   # the records are only read
    return out[0], sim.query(7) - before


@pytest.mark.parametrize("kind,n,frames", [("diff", 24, 6), ("trajopt", 40, 5), ("batching", 80, 3), ("separation", 30, 4),
                                           ("selfcontact", 60, 3)])
def test_stored_records_give_the_recomputed_gradients(kind, n, frames):
    p = inputs.small_case(kind, n_rods=4, n=n, frames=frames)
    ref, launches = gradients(p, frames, hbm_budget=1 << 20)       # too little: recompute, in chunks
    for kw in (dict(), dict(chunks=(1, frames - 1)), dict(checkpoint_every=2), dict(plain_first=True)):
        got, l2 = gradients(p, frames, **kw)
        if not kw:
            assert l2 < launches    # no recompute kernel ran
        for k in ref:
            a, b = got[k].double(), ref[k].double()
            if kind in ("selfcontact", "separation"):
                assert float((a - b).norm()) <= 1e-4 * float(b.norm()) + 1e-20, (kw, k)
            else:
                assert torch.equal(a, b), (kw, k, float((a - b).abs().max()))


def test_forced_substeps_beyond_the_planned_records():
    """Substeps forced at the step are more than the records were laid out for."""
    p = inputs.small_case("diff", n_rods=3, n=24, frames=4)
    ref, _ = gradients(p, 4, substeps=23, hbm_budget=1 << 20)
    got, _ = gradients(p, 4, substeps=23)
    for k in ref:
        assert torch.equal(got[k], ref[k]), k


def test_a_captured_step_stores_no_records():
    """The graph may outlive the records' buffer, so the backward of a captured step recomputes."""
    p = inputs.small_case("diff", n_rods=3, n=24, frames=4)
    ref, _ = gradients(p, 4, hbm_budget=1 << 20)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        sim = sim_for(p)
        wx, wv, wth = (torch.as_tensor(w, dtype=torch.float32, device="cuda") for w in weights(p, 2))
        acts = actions_dev(p)
        sim.reset()
        sim.begin_rollout(4)
        g = torch.cuda.CUDAGraph()
        stream.synchronize()
        with torch.cuda.graph(g, stream=stream, capture_error_mode="thread_local"):
            sim.step(acts, 4)
        g.replay()
        got = sim.backward(wx, wv, wth)
        stream.synchronize()
    for k in ref:
        assert torch.equal(got[k], ref[k]), k


@pytest.mark.parametrize("n", [128, 192, 224, 256])
def test_recording_changes_neither_state_nor_gradient(n):
    """Yielding wires of each size class: a hinge on its yield surface branches on the last bit of
    its curvature, so the three kernels that step a rod have to round alike."""
    p = inputs.batching(60, 1, 5, vmin=n - 31, vmax=n)
    p.E[:], p.K[:], p.G[:] = (inputs.f32(np.full(60, v)) for v in (1e5, 1e5, 4e4))
    sim = sim_for(p)
    states = []
    for record in (False, True):
        sim.reset()
        if record:
            sim.begin_rollout(1)
        sim.step(actions_dev(p), 1)
        states.append(sim.full_state_numpy())
    for k in states[0]:
        assert np.array_equal(states[0][k], states[1][k]), k
    ref, _ = gradients(p, 1, hbm_budget=1 << 20)
    got, _ = gradients(p, 1)
    for k in ref:
        assert torch.equal(got[k], ref[k]), k

"""The silhouette loss's workspace depends on the rods and the number of pixels alone, so a call held
in a CUDA graph keeps its memory when later calls ask for the gradient too, use more cameras or
another image shape; and cameras beyond one group add up as the others do."""
import math

import numpy as np
import pytest
import torch

from oracle.silhouette import camera
from paper_2606_04206_gb300 import dlo, inputs
from gpu_util import sim_for

pytestmark = pytest.mark.gpu


def rods(n_rods=3, n=40):
    s = np.linspace(0.0, 0.9, n)
    return inputs.custom([np.stack([0.3 * s - 0.15, 0.05 * np.sin(7 * s + b), 0.3 + 0.02 * np.cos(5 * s)], 1)
                          for b in range(n_rods)], K=1e5, E=1e4)


def look(n_cams, height, width, batch, seed=0):
    rng = np.random.default_rng(seed)
    cams = []
    for k in range(n_cams):
        a = 0.2 * k
        R = np.diag([1.0, -1.0, -1.0]) @ np.array([[math.cos(a), -math.sin(a), 0.0], [math.sin(a), math.cos(a), 0.0], [0.0, 0.0, 1.0]])
        f = 0.9 * max(height, width)
        cams.append(camera(f, f, width / 2, height / 2, R, [0.01 * k, 0.0, 1.2]))
    masks = (rng.uniform(size=(batch, n_cams, height, width)) < 0.3).astype(np.uint8)
    return torch.tensor(np.stack(cams), dtype=torch.float32, device="cuda"), torch.tensor(masks, device="cuda")


def test_later_calls_leave_the_workspace_where_it_is():
    calls = []

    def alloc(nbytes):
        calls.append(nbytes)
        return torch.cuda.caching_allocator_alloc(nbytes, torch.cuda.current_device(), torch.cuda.current_stream())

    sim_for(rods()).close()   # the library is built
    p = rods()
    sim = dlo.DloSim(p, allocator=(alloc, torch.cuda.caching_allocator_delete))
    x = sim.tensors_from_problem()[0]
    sim.silhouette(x, *look(1, 48, 64, p.batch), grad=False)
    before = len(calls)
    for n_cams, h, w in ((1, 48, 64), (2, 48, 64), (9, 48, 64), (1, 64, 48), (1, 3072, 1), (1, 1, 3072), (3, 7, 70), (2, 5, 3)):
        for grad in (False, True):
            sim.silhouette(x, *look(n_cams, h, w, p.batch), grad=grad, render=grad)
    assert len(calls) == before


def test_a_replayed_value_after_a_gradient_with_more_cameras():
    p = rods()
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        sim = sim_for(p)
        x = sim.tensors_from_problem()[0]
        cams, masks = look(1, 48, 64, p.batch)
        ref, _, _ = sim.silhouette(x, cams, masks, grad=False)
        stream.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream, capture_error_mode="thread_local"):
            q, _, _ = sim.silhouette(x, cams, masks, grad=False)
        sim.silhouette(x, *look(6, 48, 64, p.batch))
        other = [torch.full((1 << 16,), 7.0, device="cuda") for _ in range(8)]   # takes up freed memory
        g.replay()
        stream.synchronize()
    assert torch.equal(q, ref) and all(bool((t == 7.0).all()) for t in other)


@pytest.mark.parametrize("n_cams", [4, 5, 9])
def test_groups_of_cameras(n_cams):
    """The loss is the mean over cameras: against one call per camera, whose terms are the same up to
    the rounding of 1 / (cameras x pixels), of the sums over the cameras (n_cams x 6e-8) and of their
    mean; 2e-6 of the largest gradient.  The gradient may overwrite the positions."""
    p = rods()
    sim = sim_for(p)
    x = sim.tensors_from_problem()[0]
    cams, masks = look(n_cams, 48, 64, p.batch)
    q, gx, img = sim.silhouette(x, cams, masks, render=True)
    one = [sim.silhouette(x, cams[c:c + 1], masks[:, c:c + 1], render=True) for c in range(n_cams)]
    assert torch.equal(img, torch.cat([o[2] for o in one], 1))
    qm = torch.stack([o[0].double() for o in one]).mean(0)
    gm = torch.stack([o[1].double() for o in one]).mean(0)
    assert float((q.double() - qm).abs().max()) <= 1e-6 * float(qm.max())
    assert float((gx.double() - gm).abs().max()) <= 2e-6 * float(gm.abs().max())
    y = x.clone()
    ptr = lambda t: t.data_ptr()
    st = sim.lib.dlo_loss_silhouette(sim.ctx, ptr(y), ptr(cams), n_cams, 48, 64, ptr(masks), 1.0, None, None, ptr(y), None)
    assert st == 0
    torch.cuda.synchronize()
    assert torch.equal(y, gx)

"""Where the forward stores substep records, and whose memory they take: in the workspace that an
earlier dlo_backward of the context left, and nowhere else.  Which path ran is read from the launch
counter: a backward on stored records launches one reverse per size class and the frames' adjoint,
one that recomputes also a recompute kernel per class (one chunk holds these rollouts)."""
import numpy as np
import pytest
import torch

from paper_2606_04206_gb300 import dlo, inputs
from gpu_util import actions_dev, grad_agreement, sim_for
from test_gpu_backward import weights

pytestmark = pytest.mark.gpu


class Counting:
    """Allocations through torch, with the bytes that are out."""

    def __init__(self):
        self.size, self.live, self.on_free = {}, 0, None

    def alloc(self, nbytes):
        ptr = torch.cuda.caching_allocator_alloc(nbytes, torch.cuda.current_device(), torch.cuda.current_stream())
        self.size[ptr] = nbytes
        self.live += nbytes
        return ptr

    def free(self, ptr):
        if self.on_free:
            self.on_free()
        self.live -= self.size.pop(ptr)
        torch.cuda.caching_allocator_delete(ptr)


class Rollouts:
    def __init__(self, p, **opt):
        from paper_2606_04206_gb300 import build
        build.build()
        self.mem = Counting()
        self.p, self.sim = p, dlo.DloSim(p, allocator=(self.mem.alloc, self.mem.free), **opt)
        self.w = [torch.as_tensor(w, dtype=torch.float32, device="cuda") for w in weights(p, 2)]

    def forward(self, frames, chunks=None, substeps=0, plain=False):
        self.sim.reset()
        self.sim.begin_rollout(frames)
        f = 0
        for n in chunks or (frames,):
            before = self.sim.query(dlo.Q_LAUNCHES)
            acts = actions_dev(self.p, f, f + n)
            self.sim.step_plain(acts, n, substeps) if plain else self.sim.step(acts, n, substeps)
            self.classes = self.sim.query(dlo.Q_LAUNCHES) - before   # a step is one launch per class
            f += n

    def backward(self, recomputes):
        before = self.sim.query(dlo.Q_LAUNCHES)
        g = self.sim.backward(*self.w)
        assert self.sim.query(dlo.Q_LAUNCHES) - before == (2 if recomputes else 1) * self.classes + 1
        return g


def agree(p, got, ref):
    for k in ref:
        if p.self_contact:   # pairs are reversed with float atomics
            assert float((got[k] - ref[k]).norm()) <= 1e-4 * float(ref[k].norm()) + 1e-20, k
        else:
            assert torch.equal(got[k], ref[k]), k


@pytest.mark.parametrize("opt", [dict(), dict(checkpoint_every=2)])
@pytest.mark.parametrize("kind,n,frames", [("diff", 24, 6), ("trajopt", 40, 5), ("batching", 80, 3), ("separation", 30, 4),
                                           ("selfcontact", 60, 3)])
def test_the_second_rollout_stores_its_records(kind, n, frames, opt):
    p = inputs.small_case(kind, n_rods=4, n=n, frames=frames)
    r = Rollouts(p, **opt)
    r.forward(frames)
    ref = r.backward(recomputes=True)
    for chunks in (None, (1, frames - 1)):
        r.forward(frames, chunks)
        agree(p, r.backward(recomputes=False), ref)
        agree(p, r.backward(recomputes=False), ref)   # the records are only read


def test_what_cannot_be_stored_is_recomputed_in_the_same_memory():
    """After a rollout of 4 frames: a longer one, more substeps than the workspace holds, plain
    steps, a plain backward in between, a shorter one.  No way needs more than its own
    recomputation, and each gradient is that of a context that has only recomputed."""
    p = inputs.small_case("diff", n_rods=3, n=24, frames=6)

    def fresh(frames, **kw):
        r = Rollouts(p)
        r.forward(frames, **kw)
        return r.backward(recomputes=True), r.mem.live

    r = Rollouts(p)
    r.forward(4)
    r.backward(recomputes=True)
    for frames, kw in ((6, {}), (4, dict(substeps=23))):
        r.forward(frames, **kw)
        ref, live = fresh(frames, **kw)
        agree(p, r.backward(recomputes=True), ref)
    most = r.mem.live
    assert most <= live + r.sim.B * 96 * 6 + 16 * 6 * (3 * r.sim.V + 2 * r.sim.E)   # the ring and actions of 6 frames
    ref, _ = fresh(4)
    r.forward(4)
    agree(p, r.backward(recomputes=False), ref)
    plain = r.sim.backward(*r.w, plain=True)   # takes over the workspace the records are in
    for k in ref:
        rel, cos = grad_agreement(plain[k].double().cpu().numpy(), ref[k].double().cpu().numpy())
        assert rel <= 1e-3 and cos >= 0.999, k
    most = r.mem.live   # with the plain kernels' own scratch
    agree(p, r.backward(recomputes=True), ref)
    r.forward(4)
    agree(p, r.backward(recomputes=False), ref)
    r.forward(4, plain=True)
    r.classes = 1
    got = r.backward(recomputes=True)
    for k in ref:
        rel, cos = grad_agreement(got[k].double().cpu().numpy(), ref[k].double().cpu().numpy())
        assert rel <= 1e-3 and cos >= 0.999, k
    assert r.mem.live == most


def test_a_captured_step_takes_no_second_workspace():
    p = inputs.small_case("diff", n_rods=3, n=24, frames=4)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        r = Rollouts(p)
        r.forward(4)
        ref = r.backward(recomputes=True)
        live, acts = r.mem.live, actions_dev(p)
        r.sim.reset()
        r.sim.begin_rollout(4)
        stream.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream, capture_error_mode="thread_local"):
            r.sim.step(acts, 4)
        g.replay()
        got = r.backward(recomputes=True)
        stream.synchronize()
    agree(p, got, ref)
    assert r.mem.live == live


@pytest.mark.parametrize("how", ["noalloc", "plain"])
def test_other_backwards_hold_and_write_no_records(how):
    """A caller of dlo_backward_noalloc (or the plain comparator) has the ring and the action record
    from dlo_begin_rollout, and no substep records."""
    p = inputs.small_case("trajopt", n_rods=4, n=40, frames=5)
    r = Rollouts(p)
    B, V, E, F = p.batch, r.sim.V, r.sim.E, 5
    before = r.mem.live
    for _ in range(2):
        r.forward(F)
        ring = F * (16 * (3 * V + 2 * E) + 96 * B) + 8 * 256
        assert r.mem.live - before <= ring + 48 * B * F + 2 * 256 or how == "plain"
        out = r.sim.backward_noalloc(*r.w) if how == "noalloc" else r.sim.backward(*r.w, plain=True)
    # back to dlo_backward: it recomputes once more, then finds its records stored
    ref = r.backward(recomputes=True)
    r.forward(F)
    agree(p, r.backward(recomputes=False), ref)
    if how == "noalloc":
        r.sim.backward_noalloc(*r.w)
        r.forward(F)
        agree(p, r.backward(recomputes=True), ref)   # nothing was stored for the call that reads nothing
    for k in out:
        rel, cos = grad_agreement(out[k].double().cpu().numpy(), ref[k].double().cpu().numpy())
        assert rel <= 1e-3 and cos >= 0.999, k


def test_the_workspace_is_given_back_when_nothing_writes_it():
    """A rollout that stores its records and is abandoned, then a longer one whose backward needs a
    larger workspace: the old one goes back to the caller's allocator after the steps have ended."""
    p = inputs.small_case("diff", n_rods=1500, n=60, frames=8)
    r = Rollouts(p)
    r.forward(4)
    r.backward(recomputes=True)
    r.sim.begin_rollout(4)
    r.sim.step(actions_dev(p, 0, 4), 4)
    r.sim.begin_rollout(8)
    acts, busy = actions_dev(p), []
    r.mem.on_free = lambda: busy.append(not torch.cuda.current_stream().query())
    r.sim.step(acts, 8)
    r.sim.backward(*r.w)
    r.mem.on_free = None
    assert busy == [False]

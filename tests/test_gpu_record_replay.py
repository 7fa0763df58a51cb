"""The gradient of a rollout replayed from a CUDA graph, after the same context has differentiated
another one step by step: a replay writes the checkpoints and the actions anew, and the backward
that follows is the replayed rollout's."""
import pytest
import torch

from paper_2606_04206_gb300 import inputs
from gpu_util import actions_dev, sim_for
from test_gpu_backward import weights

pytestmark = pytest.mark.gpu


def test_replay_after_an_eager_rollout():
    p = inputs.small_case("diff", n_rods=3, n=24, frames=4)
    acts = actions_dev(p)
    other = (acts * -0.5 + 1e-4).contiguous()
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        sim = sim_for(p)
        state = sim.tensors_from_problem()
        w = [torch.as_tensor(a, dtype=torch.float32, device="cuda") for a in weights(p, 2)]

        def forward(a):
            sim.set_state(*state)
            sim.begin_rollout(4)
            sim.step(a, 4)

        def eager():
            forward(acts)
            return sim.backward(*w)

        forward(other)
        ref = sim.backward(*w)
        first = [eager() for _ in range(2)]     # the second may find its records stored
        buf = other.clone()
        stream.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream, capture_error_mode="thread_local"):
            forward(buf)
        g.replay()
        replayed = sim.backward(*w)
        again = eager()
        g.replay()
        after = sim.backward(*w)
        stream.synchronize()
    for k in ref:
        assert torch.equal(first[0][k], first[1][k]) and torch.equal(again[k], first[0][k]), k
        assert torch.equal(replayed[k], ref[k]), k
        assert torch.equal(after[k], ref[k]), k
    assert not torch.equal(ref["actions"], first[0]["actions"])

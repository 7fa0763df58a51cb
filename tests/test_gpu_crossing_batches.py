"""A rod's crossing loss and gradient are the same alone and in a batch with shorter or longer ones."""
import numpy as np
import pytest
import torch

from paper_2606_04206_gb300 import dlo, inputs
from gpu_util import sim_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [(40, 128, 129, 256), (8, 200), (127, 129)])
def test_alone_and_in_a_batch(sizes):
    rods = []
    for n in sizes:
        s = np.linspace(0.0, 1.8 * np.pi, n)
        rods.append(0.06 * np.stack([np.sin(s) + 2 * np.sin(2 * s), np.cos(s) - 2 * np.cos(2 * s), -np.sin(3 * s)], 1)
                    + [0.0, 0.0, 0.3])
    p = inputs.custom(rods, K=1e5, E=1e4)
    sim = sim_for(p)
    q, gx = sim.loss(dlo.LOSS_CROSSING, sim.tensors_from_problem()[0])
    for b, rod in enumerate(rods):
        one = sim_for(inputs.custom([rod], K=1e5, E=1e4))
        q1, g1 = one.loss(dlo.LOSS_CROSSING, one.tensors_from_problem()[0])
        assert torch.equal(q[b:b + 1], q1) and torch.equal(gx[p.vert_off[b]:p.vert_off[b + 1]], g1), b

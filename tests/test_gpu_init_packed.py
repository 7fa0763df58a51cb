"""Initial frames and states of short rods in large batches, several rods to a warp, against the
same rods in a small batch, a block each: bit for bit, for every size up to a warp, open rods, loops
and strands, at every packing, alone and beside longer rods."""
import numpy as np
import pytest
import torch

from paper_2606_04206_gb300 import inputs
from gpu_util import sim_for
from test_gpu_init_frames import curve

pytestmark = pytest.mark.gpu


def problem(sizes, seed):
    rng = np.random.default_rng(seed)
    rods, closed, cut = [], [], []
    for n in sizes:
        for kind in range(3):   # open, loop, two strands
            loop = kind == 1 and n >= 3
            rods.append(curve(rng, n, loop))
            closed.append(loop)
            cut.append(n // 2 if kind == 2 and n >= 4 else 0)
    p = inputs.custom(rods, closed=closed, K=0.0, E=1e4, G=1e3, inextensible=True)
    for b, c in enumerate(cut):
        if c:
            p.strand_start[p.vert_off[b] + c] = True
    p.theta0[:] = inputs.f32(rng.normal(size=p.theta0.shape))
    p.v0[:] = inputs.f32(rng.normal(size=p.v0.shape))
    return p


@pytest.mark.parametrize("sizes", [(2, 3, 4), (2, 5, 8), (3, 9, 16), (2, 16, 33, 130), (4, 17, 31, 32, 200)])
def test_packed_equals_a_block_per_rod(sizes):
    few = problem(sizes, len(sizes))
    order = np.random.default_rng(0).integers(0, few.batch, 6001)
    many = few.subset(order)
    a, b = sim_for(few), sim_for(many)
    for rest in (True, False):   # the state of dlo_create, then of dlo_set_state
        if not rest:
            a.reset()
            b.reset()
        sa, sb = a.full_state_numpy(), b.full_state_numpy()
        for k in sa:
            per = sa[k]
            if k in ("x", "v", "kbar", "mprev", "mbar"):
                per = np.concatenate([per[few.vert_off[r]:few.vert_off[r + 1]] for r in order])
            elif k in ("theta", "omega", "d1b", "tb"):
                per = np.concatenate([per[few.edge_off[r]:few.edge_off[r + 1]] for r in order])
            else:
                per = per[order]
            assert np.array_equal(per, sb[k]), (rest, k)

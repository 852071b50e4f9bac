"""The two tile shapes of the FP64 3-D WENO-Z kernels, 32 x 8 and 32 x 4 (the
context takes the one with the shorter launch): grids at the edges of both
against the FP64 oracle at the tolerance of every FP64 comparison (1e-12 relative
L1 per variable), and bit for bit against each other: a periodic (32, 64, 4) grid
(eight 32 x 8 tiles leave most SMs idle: 32 x 4) and its 19-fold repetition in x
(152 tiles of 32 x 8) evolve the same cells."""
import numpy as np
import pytest

import oracle as orc
from paper_2510_24175_gb300.inputs import Problem
from parity_util import gpu_run, oracle_run, rel_l1

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(31, 3, 3), (32, 4, 5), (33, 8, 4), (65, 9, 7)])
@pytest.mark.parametrize("rk,bc", [(3, (0,) * 6), (2, (1,) * 6)])
def test_wenoz_tile_edges(n, rk, bc):
    pb = Problem("random_smooth", n, seed=8, limiter=orc.LIM_WENOZ, rk_order=rk, bc=bc)
    ref = oracle_run(pb, 2)
    U, _, cnt = gpu_run(pb, 2)
    assert cnt == {"rho_floor": 0, "p_floor": 0, "status": 0, "p_f64": 0}
    err = rel_l1(U, ref.U)
    assert np.all(err <= 1e-12), err


def test_wenoz_tile_shapes_agree_bit_for_bit():
    import torch
    import paper_2510_24175_gb300 as m
    V = torch.from_numpy(Problem("random_smooth", (32, 64, 4), seed=3).prim()).cuda()
    out = []
    for reps in (1, 19):
        prim = V.repeat(1, 1, 1, reps).contiguous()
        s = m.MHD(m.Config(n=tuple(prim.shape[:0:-1]), dx=(1.0 / 32,) * 3, rk_order=3,
                           limiter=orc.LIM_WENOZ))
        s.set_state(prim, kind=m.MHD_PRIM)
        for _ in range(2):
            s.step()
        out.append(s.get_state())
    assert torch.equal(out[1], out[0].repeat(1, 1, 1, 19))

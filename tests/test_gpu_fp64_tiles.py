"""The two tile shapes of the FP64 3-D PLM kernels, 32 x 8 and 16 x 16 (the context
takes the one with the shorter launch): grids at the edges of both against the
FP64 oracle at the tolerance of every FP64 comparison (1e-12 relative L1 per
variable), and bit for bit against each other: a periodic (32, 8, nz) grid (32 x 8
tiles; 16 x 16 would be half empty) and its doubling in y (16 x 16 tiles) evolve
the same cells."""
import numpy as np
import pytest

import oracle as orc
from paper_2510_24175_gb300.inputs import Problem
from parity_util import gpu_run, oracle_run, rel_l1

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(15, 15, 2), (16, 16, 3), (17, 17, 7), (33, 31, 5), (48, 49, 9)])
@pytest.mark.parametrize("limiter,bc", [(orc.LIM_MC, (0,) * 6), (orc.LIM_MINMOD, (1,) * 6)])
def test_fp64_tile_edges(n, limiter, bc):
    pb = Problem("random_smooth", n, seed=5, limiter=limiter, bc=bc)
    ref = oracle_run(pb, 2)
    U, _, cnt = gpu_run(pb, 2)
    assert cnt == {"rho_floor": 0, "p_floor": 0, "status": 0, "p_f64": 0}
    err = rel_l1(U, ref.U)
    assert np.all(err <= 1e-12), err


@pytest.mark.parametrize("nz", [4, 11])
@pytest.mark.parametrize("rk", [2, 3])
def test_tile_shapes_agree_bit_for_bit(nz, rk):
    import torch
    import paper_2510_24175_gb300 as m
    V = torch.from_numpy(Problem("random_smooth", (32, 8, nz), seed=3).prim()).cuda()
    out = []
    for prim in (V, torch.cat((V, V), dim=2).contiguous()):
        n = tuple(prim.shape[:0:-1])
        s = m.MHD(m.Config(n=n, dx=(1.0 / 32,) * 3, rk_order=rk))
        s.set_state(prim, kind=m.MHD_PRIM)
        for _ in range(3):
            s.step()
        out.append(s.get_state())
    one, two = out
    assert torch.equal(two[:, :, :8], one) and torch.equal(two[:, :, 8:], one)

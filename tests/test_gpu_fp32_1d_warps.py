"""1-D FP32 grids on either side of the line between two warps and one per tile
(4 tiles per SM): the grids next to it against the FP64 oracle at the FP32 bound of
the other comparisons (2e-5 relative L1 per variable, the norm's floor at 0.1
||rho||_1), and a periodic grid of two-warp tiles bit for bit against its
repetition, which takes one warp."""
import numpy as np
import pytest

import oracle as orc
from paper_2510_24175_gb300.inputs import Problem
from parity_util import gpu_run, oracle_run, rel_l1

pytestmark = pytest.mark.gpu


def warps(cfg):
    import torch
    import paper_2510_24175_gb300 as m
    return m.mhd_plan_stage(cfg.c(),
                            torch.cuda.get_device_properties(0).multi_processor_count)["warps"]


@pytest.mark.parametrize("beyond,nw", [(-1, 2), (0, 2), (1, 1), (33, 1)])
@pytest.mark.parametrize("limiter,rk,bc", [(orc.LIM_MC, 2, 0), (orc.LIM_MINMOD, 3, 1),
                                           (orc.LIM_WENOZ, 3, 0)])
def test_grids_next_to_the_line(beyond, nw, limiter, rk, bc):
    import torch
    import paper_2510_24175_gb300 as m
    n = 32 * 4 * torch.cuda.get_device_properties(0).multi_processor_count + beyond
    pb = Problem("random_smooth", (n, 1, 1), seed=6, limiter=limiter, rk_order=rk, bc=(bc,) * 6)
    assert warps(m.Config.from_problem(pb, precision=m.MHD_FP32)) == nw
    ref = oracle_run(pb, 2)
    U, _, cnt = gpu_run(pb, 2, precision=m.MHD_FP32)
    assert cnt["status"] == 0
    err = rel_l1(U, ref.U, floor=0.1)
    assert np.all(err <= 2e-5), err


@pytest.mark.parametrize("limiter,rk", [(orc.LIM_MC, 2), (orc.LIM_FLAT, 3), (orc.LIM_WENOZ, 3)])
def test_one_and_two_warps_agree_bit_for_bit(limiter, rk):
    import torch
    import paper_2510_24175_gb300 as m
    V = torch.from_numpy(Problem("random_smooth", (9600, 1, 1), seed=3).prim()).cuda()
    reps = 4 * torch.cuda.get_device_properties(0).multi_processor_count // 300 + 1
    out = []
    for prim, nw in ((V, 2), (V.repeat(1, 1, 1, reps).contiguous(), 1)):
        cfg = m.Config(n=tuple(prim.shape[:0:-1]), dx=(1.0 / 32,) * 3, rk_order=rk,
                       limiter=limiter, precision=m.MHD_FP32)
        assert warps(cfg) == nw
        s = m.MHD(cfg)
        s.set_state(prim, kind=m.MHD_PRIM)
        for _ in range(5):
            s.step()
        out.append(s.get_state())
    assert torch.equal(out[1], out[0].repeat(1, 1, 1, reps))

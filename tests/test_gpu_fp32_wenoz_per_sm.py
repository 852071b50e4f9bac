"""The two forms of the FP32 3-D WENO-Z kernels, one CTA per SM and two (the plan
takes one where a launch does not need the second slot), each test asserting the
planned form: ragged grids with cleaning against the FP64 oracle at the FP32 bound of the other
comparisons (2e-5 relative L1 per variable, the norm's floor at 0.1 ||rho||_1); bit
for bit against each other, by a periodic repetition that plans the other one,
with cleaning and with constrained transport; and blocks with halo faces."""
import numpy as np
import pytest

import oracle as orc
from paper_2510_24175_gb300 import inputs
from paper_2510_24175_gb300.inputs import Problem
from parity_util import gpu_run, oracle_run, rel_l1

pytestmark = pytest.mark.gpu


def per_sm(cfg):
    import torch
    import paper_2510_24175_gb300 as m
    return m.mhd_plan_stage(
        cfg.c(), torch.cuda.get_device_properties(0).multi_processor_count)["ctas_per_sm"]


@pytest.mark.parametrize("n,k", [((33, 9, 200), 2), ((40, 33, 75), 2), ((99, 9, 100), 2),
                                 ((33, 18, 300), 1), ((31, 7, 5), 1)])
@pytest.mark.parametrize("rk,bc", [(3, (0,) * 6), (2, (1,) * 6)])
def test_ragged_grids(n, k, rk, bc):
    import paper_2510_24175_gb300 as m
    pb = Problem("random_smooth", n, seed=8, bc=bc, limiter=orc.LIM_WENOZ, rk_order=rk)
    assert per_sm(m.Config.from_problem(pb, precision=m.MHD_FP32)) == k
    ref = oracle_run(pb, 2)
    U, _, cnt = gpu_run(pb, 2, precision=m.MHD_FP32)
    assert cnt["status"] == 0
    err = rel_l1(U, ref.U, floor=0.1)
    assert np.all(err <= 2e-5), err


@pytest.mark.parametrize("divb", [0, 1])
def test_forms_agree_bit_for_bit(divb):
    import torch
    import paper_2510_24175_gb300 as m
    n = (33, 9, 100)
    pb = inputs.ct_random(n, seed=3) if divb else Problem("random_smooth", n, seed=3)
    out = []
    for k in (1, 2):
        V = torch.from_numpy(pb.prim()).cuda().repeat(1, k, 1, 1).contiguous()
        cfg = m.Config(n=tuple(V.shape[:0:-1]), dx=(1.0 / 32,) * 3, rk_order=3,
                       limiter=orc.LIM_WENOZ, precision=m.MHD_FP32, divb=pb.divb)
        assert per_sm(cfg) == k
        s = m.MHD(cfg)
        s.set_state(V, kind=m.MHD_PRIM)
        if divb:
            s.set_face_field(torch.from_numpy(pb.faces()).cuda().repeat(1, k, 1, 1).contiguous())
        for _ in range(2):
            s.step()
        out.append(s.get_state())
    assert torch.equal(out[1], out[0].repeat(1, 2, 1, 1))


@pytest.mark.parametrize("n,whole,block", [((33, 9, 200), 2, 1), ((33, 37, 240), 2, 2)])
@pytest.mark.parametrize("bc", [(0,) * 6, (1,) * 6])
def test_blocks_with_halo_faces(n, whole, block, bc):
    import torch
    import paper_2510_24175_gb300 as m
    from paper_2510_24175_gb300.decomp import LocalBlocks
    pb = Problem("random_smooth", n, seed=29, bc=bc, limiter=orc.LIM_WENOZ, rk_order=3)
    cfg = m.Config.from_problem(pb, precision=m.MHD_FP32)
    V = torch.from_numpy(pb.prim()).cuda()
    s = m.MHD(cfg)
    lb = LocalBlocks(cfg, (1, 1, 2))
    assert per_sm(cfg) == whole and {per_sm(b.config) for b in lb.blocks} == {block}
    for x in (s, lb):
        x.set_state(V, kind=m.MHD_PRIM)
        for _ in range(2):
            x.step()
    assert torch.equal(lb.get_state(), s.get_state())

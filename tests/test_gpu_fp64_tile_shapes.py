"""FP64 3-D PLM grids whose plan is the 32 x 8 column tile (most plan 16 x 16), each
test asserting the planned shapes: ragged edges against the FP64 oracle at the
tolerance of every FP64 comparison (1e-12 relative L1 per variable); bit for bit
against 16 x 16 tiles, by a periodic repetition that plans those; and
decompositions in which the blocks and the whole grid take different shapes."""
import numpy as np
import pytest

import oracle as orc
from paper_2510_24175_gb300.inputs import Problem
from parity_util import gpu_run, oracle_run, rel_l1

pytestmark = pytest.mark.gpu


def tile(cfg):
    import torch
    import paper_2510_24175_gb300 as m
    p = m.mhd_plan_stage(cfg.c(), torch.cuda.get_device_properties(0).multi_processor_count)
    return p["tx"], p["ty"]


@pytest.mark.parametrize("n", [(37, 4, 202), (33, 5, 216), (26, 37, 103), (151, 5, 72)])
@pytest.mark.parametrize("limiter,bc", [(orc.LIM_MC, (0,) * 6), (orc.LIM_MINMOD, (1,) * 6)])
def test_ragged_32x8_tiles(n, limiter, bc):
    import paper_2510_24175_gb300 as m
    pb = Problem("random_smooth", n, seed=5, limiter=limiter, bc=bc)
    assert tile(m.Config.from_problem(pb)) == (32, 8)
    ref = oracle_run(pb, 2)
    U, _, cnt = gpu_run(pb, 2)
    assert cnt == {"rho_floor": 0, "p_floor": 0, "status": 0, "p_f64": 0}
    err = rel_l1(U, ref.U)
    assert np.all(err <= 1e-12), err


@pytest.mark.parametrize("n,reps", [((37, 4, 202), (1, 1, 3, 1)), ((33, 5, 216), (1, 1, 1, 2))])
@pytest.mark.parametrize("rk", [2, 3])
def test_shapes_agree_bit_for_bit(n, reps, rk):
    import torch
    import paper_2510_24175_gb300 as m
    V = torch.from_numpy(Problem("random_smooth", n, seed=3).prim()).cuda()
    out = []
    for prim, shape in ((V, (32, 8)), (V.repeat(*reps).contiguous(), (16, 16))):
        cfg = m.Config(n=tuple(prim.shape[:0:-1]), dx=(1.0 / 32,) * 3, rk_order=rk)
        assert tile(cfg) == shape
        s = m.MHD(cfg)
        s.set_state(prim, kind=m.MHD_PRIM)
        for _ in range(3):
            s.step()
        out.append(s.get_state())
    assert torch.equal(out[1], out[0].repeat(*reps))


@pytest.mark.parametrize("n,dims,whole,block", [
    ((37, 4, 202), (1, 1, 2), (32, 8), (16, 16)), ((33, 10, 216), (1, 2, 1), (16, 16), (32, 8)),
    ((52, 37, 103), (2, 1, 1), (32, 8), (32, 8))])
@pytest.mark.parametrize("bc", [(0,) * 6, (1,) * 6])
def test_blocks_of_another_shape(n, dims, whole, block, bc):
    import torch
    import paper_2510_24175_gb300 as m
    from paper_2510_24175_gb300.decomp import LocalBlocks
    pb = Problem("random_smooth", n, seed=29, bc=bc)
    cfg = m.Config.from_problem(pb)
    V = torch.from_numpy(pb.prim()).cuda()
    s = m.MHD(cfg)
    lb = LocalBlocks(cfg, dims)
    assert tile(cfg) == whole and {tile(b.config) for b in lb.blocks} == {block}
    for x in (s, lb):
        x.set_state(V, kind=m.MHD_PRIM)
        for _ in range(3):
            x.step()
    assert torch.equal(lb.get_state(), s.get_state())

"""FP64 3-D WENO-Z grids whose plan is the 32 x 8 column tile (small grids plan 32 x
4), each test asserting the planned shapes: ragged edges against the FP64 oracle
at the tolerance of every FP64 comparison (1e-12 relative L1 per variable), with
cleaning and with constrained transport; bit for bit against 32 x 4 tiles, by a
periodic repetition that plans those; and blocks with halo faces."""
import numpy as np
import pytest

import oracle as orc
from paper_2510_24175_gb300 import inputs
from paper_2510_24175_gb300.inputs import Problem
from parity_util import gpu_run, oracle_run, rel_l1
from test_gpu_fp64_tile_shapes import tile

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(4, 26, 268), (7, 217, 20), (33, 37, 120)])
@pytest.mark.parametrize("rk,bc,divb", [(3, (0,) * 6, 0), (2, (1,) * 6, 0), (3, (0,) * 6, 1)])
def test_ragged_32x8_tiles(n, rk, bc, divb):
    import paper_2510_24175_gb300 as m
    pb = inputs.ct_random(n, seed=8) if divb else Problem("random_smooth", n, seed=8, bc=bc)
    pb.limiter, pb.rk_order = orc.LIM_WENOZ, rk
    assert tile(m.Config.from_problem(pb)) == (32, 8)
    ref = oracle_run(pb, 2)
    U, _, cnt = gpu_run(pb, 2)
    assert cnt == {"rho_floor": 0, "p_floor": 0, "status": 0, "p_f64": 0}
    err = rel_l1(U, ref.U)
    assert np.all(err <= 1e-12), err


@pytest.mark.parametrize("n,reps", [((33, 37, 120), (1, 1, 2, 1)), ((7, 217, 20), (1, 1, 1, 5))])
def test_shapes_agree_bit_for_bit(n, reps):
    import torch
    import paper_2510_24175_gb300 as m
    V = torch.from_numpy(Problem("random_smooth", n, seed=3).prim()).cuda()
    out = []
    for prim, shape in ((V, (32, 8)), (V.repeat(*reps).contiguous(), (32, 4))):
        cfg = m.Config(n=tuple(prim.shape[:0:-1]), dx=(1.0 / 32,) * 3, rk_order=3,
                       limiter=orc.LIM_WENOZ)
        assert tile(cfg) == shape
        s = m.MHD(cfg)
        s.set_state(prim, kind=m.MHD_PRIM)
        for _ in range(2):
            s.step()
        out.append(s.get_state())
    assert torch.equal(out[1], out[0].repeat(*reps))


@pytest.mark.parametrize("n,dims,whole,block", [((33, 37, 240), (1, 1, 2), (32, 8), (32, 8)),
                                                ((4, 26, 268), (1, 1, 2), (32, 8), (32, 4))])
@pytest.mark.parametrize("bc", [(0,) * 6, (1,) * 6])
def test_blocks_with_halo_faces(n, dims, whole, block, bc):
    import torch
    import paper_2510_24175_gb300 as m
    from paper_2510_24175_gb300.decomp import LocalBlocks
    pb = Problem("random_smooth", n, seed=29, bc=bc, limiter=orc.LIM_WENOZ, rk_order=3)
    cfg = m.Config.from_problem(pb)
    V = torch.from_numpy(pb.prim()).cuda()
    s = m.MHD(cfg)
    lb = LocalBlocks(cfg, dims)
    assert tile(cfg) == whole and {tile(b.config) for b in lb.blocks} == {block}
    for x in (s, lb):
        x.set_state(V, kind=m.MHD_PRIM)
        for _ in range(2):
            x.step()
    assert torch.equal(lb.get_state(), s.get_state())

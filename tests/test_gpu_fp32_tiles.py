"""The FP32 3-D stage kernels at the edges of their 32 x 8 column tiles: grids one
cell short of, equal to and one cell beyond a tile, a last tile of one column
or row, few planes, against the FP64 oracle.  Tolerance: the FP32 bound of the
other comparisons with the oracle, 2e-5 relative L1 per variable with the norm's
floor at 0.1 ||rho||_1 (FP32 rounding 6e-8 amplified by two steps of smooth
flow)."""
import numpy as np
import pytest

import oracle as orc
from paper_2510_24175_gb300.inputs import Problem
from parity_util import gpu_run, oracle_run, rel_l1

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(31, 7, 4), (32, 8, 8), (33, 9, 5), (65, 17, 7), (4, 4, 4)])
@pytest.mark.parametrize("limiter,rk", [(orc.LIM_FLAT, 2), (orc.LIM_MINMOD, 2), (orc.LIM_MC, 3),
                                        (orc.LIM_WENOZ, 3)])
@pytest.mark.parametrize("bc", [(0,) * 6, (1, 1, 0, 0, 1, 1)])
def test_fp32_tile_edges(n, limiter, rk, bc):
    pb = Problem("random_smooth", n, seed=12, limiter=limiter, rk_order=rk, bc=bc)
    ref = oracle_run(pb, 2)
    U, hist, cnt = gpu_run(pb, 2, precision=1)
    assert cnt["rho_floor"] == 0 and cnt["p_floor"] == 0 and cnt["status"] == 0
    err = rel_l1(U, ref.U, floor=0.1)
    assert np.all(err <= 2e-5), err

"""Wave speeds at the ends of the number range.  States scaled by powers of two
(density s, velocity c, pressure s c^2, B c sqrt(s)) evolve as the scaled states of
scale 1, so scale 1 is the reference wherever the squares of the fast speeds are
representable (FP32: exactly; FP64, whose reciprocals and roots round differently
beyond 2^959, within the 1e-12 relative L1 of every FP64 comparison); where they
are not the step reports MHD_ERR_NONFINITE and does not return a wrong state."""
import numpy as np
import pytest

from paper_2510_24175_gb300.inputs import Problem
from parity_util import rel_l1

pytestmark = pytest.mark.gpu

GRIDS = [(64, 1, 1), (40, 24, 1), (24, 20, 12)]


def run(n, precision, limiter, s_exp, c_exp):
    import torch
    import paper_2510_24175_gb300 as m
    pb = Problem("random_smooth", n, seed=5, limiter=limiter)
    s, c, b = 2.0 ** s_exp, 2.0 ** c_exp, 2.0 ** (s_exp // 2 + c_exp)
    V = pb.prim()
    scale = np.array([s, c, c, c, b, b, b, s * c * c, b * c])[:, None, None, None]
    cfg = m.Config.from_problem(pb, precision=precision)
    cfg.rho_floor, cfg.p_floor = pb.rho_floor * s, pb.p_floor * s * c * c
    ctx = m.MHD(cfg)
    ctx.set_state(torch.from_numpy(V * scale).cuda(), kind=m.MHD_PRIM)
    for _ in range(2):
        ctx.step()
    ctx.step_info()  # raises where the device flagged the step
    scale[1:4] *= s
    return ctx.get_state().cpu().numpy() / scale


@pytest.mark.parametrize("n", GRIDS)
@pytest.mark.parametrize("precision,c_exp", [(1, 33), (1, 38), (1, 40), (0, 264), (0, 280)])
@pytest.mark.parametrize("limiter", [2, 3])
def test_speeds_whose_squares_overflow_are_reported(n, precision, c_exp, limiter):
    import paper_2510_24175_gb300 as m
    with pytest.raises(m.MHDError) as e:
        run(n, precision, limiter, 0, c_exp)
    assert e.value.code == m.MHD_ERR_NONFINITE


@pytest.mark.parametrize("n", GRIDS)
@pytest.mark.parametrize("precision,c_exp", [(1, 20), (1, 28), (0, 250), (0, -250)])
def test_speeds_inside_the_range(n, precision, c_exp):
    U, ref = run(n, precision, 2, 0, c_exp), run(n, precision, 2, 0, 0)
    assert np.all(rel_l1(U, ref) <= (0.0 if precision else 1e-12)), rel_l1(U, ref)

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


@pytest.mark.parametrize("n", GRIDS)
@pytest.mark.parametrize("s_exp,c_exp", [(40, -30), (40, -32), (40, -33), (20, -28)])
def test_fp32_speeds_with_subnormal_squares(n, s_exp, c_exp):
    """At 2^-33 and speeds of order 1 the square a^2 keeps 15 of its 24 bits or more:
    3e-5 of c_f^2, 1.5e-5 of the time step, and the two steps change the state by a
    fraction of itself: the FP32 bound 2e-5 of the other comparisons."""
    U, ref = run(n, 1, 2, s_exp, c_exp), run(n, 1, 2, 0, 0)
    assert np.all(rel_l1(U, ref, floor=0.1) <= 2e-5), rel_l1(U, ref, floor=0.1)


@pytest.mark.parametrize("n", GRIDS)
@pytest.mark.parametrize("precision,s_exp,c_exp", [(1, 0, -38), (1, 40, -38), (1, 40, -44),
                                                   (0, 0, -266), (0, 0, -280)])
def test_speeds_whose_squares_underflow_are_reported(n, precision, s_exp, c_exp):
    import paper_2510_24175_gb300 as m
    with pytest.raises(m.MHDError) as e:
        run(n, precision, 2, s_exp, c_exp)
    assert e.value.code == m.MHD_ERR_NONFINITE


def test_ensemble_boxes_report_the_range():
    import torch
    import paper_2510_24175_gb300 as m
    pb = Problem("random_smooth", (16, 12, 8), seed=5)
    scales = [2.0 ** -38, 1.0, 2.0 ** 38]
    configs = [m.Config.from_problem(pb, precision=m.MHD_FP32) for _ in scales]
    for cfg, c in zip(configs, scales):
        cfg.p_floor *= c * c
    ens = m.Ensemble(configs)
    for b, c in enumerate(scales):
        V = pb.prim()
        V[1:7] *= c
        V[7] *= c * c
        ens.set_state(b, torch.from_numpy(V).cuda(), kind=m.MHD_PRIM)
    ens.step(2)
    ens.info(1)
    for b in (0, 2):
        with pytest.raises(m.MHDError) as e:
            ens.info(b)
        assert e.value.code == m.MHD_ERR_NONFINITE

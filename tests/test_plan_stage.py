"""The plan of a context's stage launches (mhd_plan_stage, host only: the plan that
mhd_create takes) against a plain simulation of every tile shape it may choose,
and the shapes of grids that the tile tests rely on."""
import random

import pytest

import paper_2510_24175_gb300 as m
from test_plan import CANDIDATES, simulate

# (precision, limiter, divb) -> [(tx, ty, depths, weight, warps, CTAs per SM)], the first the default
MC, WZ = m.MHD_LIM_MC, m.MHD_LIM_WENOZ
SHAPES = {
    (m.MHD_FP64, MC, m.MHD_DIVB_GLM): [(32, 8, CANDIDATES, 1.0, 16, 1),
                                       (16, 16, CANDIDATES + [3, 2], 1.0, 16, 1)],
    (m.MHD_FP64, MC, m.MHD_DIVB_CT): [(32, 8, CANDIDATES, 1.0, 16, 1)],
    (m.MHD_FP64, WZ, m.MHD_DIVB_GLM): [(32, 8, CANDIDATES, 1.0, 12, 1),
                                       (32, 4, CANDIDATES, 0.54, 8, 1)],
    (m.MHD_FP64, WZ, m.MHD_DIVB_CT): [(32, 8, CANDIDATES, 1.0, 12, 1),
                                      (32, 4, CANDIDATES, 0.54, 8, 1)],
    (m.MHD_FP32, MC, m.MHD_DIVB_GLM): [(32, 8, CANDIDATES, 1.0, 16, 2)],
    (m.MHD_FP32, MC, m.MHD_DIVB_CT): [(32, 8, CANDIDATES, 1.0, 16, 2)],
    (m.MHD_FP32, WZ, m.MHD_DIVB_GLM): [(32, 8, CANDIDATES, 1.0, 16, 2),
                                       (32, 8, CANDIDATES, 0.59, 16, 1)],
    (m.MHD_FP32, WZ, m.MHD_DIVB_CT): [(32, 8, CANDIDATES, 1.0, 16, 2),
                                      (32, 8, CANDIDATES, 0.59, 16, 1)],
}


def expected(n, shapes, nsm):
    best = None
    for tx, ty, depths, weight, warps, per_sm in shapes:
        cols = -(-n[0] // tx) * -(-n[1] // ty)
        span, tz = min((simulate(cols, n[2], tz, nsm * per_sm), -tz) for tz in depths
                       if tz <= n[2] or tz == 4)
        # a later shape is taken when its launch is no longer
        if best is None or weight * span <= best[0] * best[1]["span"]:
            best = weight, {"tx": tx, "ty": ty, "tz": -tz, "warps": warps,
                            "ctas_per_sm": per_sm, "span": span}
    return best[1]


@pytest.mark.parametrize("key", sorted(SHAPES))
def test_plan_is_the_shortest_simulated_launch(key):
    rng = random.Random(11)
    taken = set()
    for _ in range(40):
        n = (rng.randint(4, 300), rng.randint(4, 200), rng.randint(4, 200))
        nsm = rng.choice([152, 152, 148, 20])
        cfg = m.Config(n=n, precision=key[0], limiter=key[1], divb=key[2]).c()
        got = m.mhd_plan_stage(cfg, nsm)
        assert got == expected(n, SHAPES[key], nsm), (n, nsm)
        taken.add((got["tx"], got["ty"], got["ctas_per_sm"]))
    assert taken == {s[:2] + s[5:] for s in SHAPES[key]}


@pytest.mark.parametrize("n,limiter,prec,tile", [
    ((256, 256, 256), MC, m.MHD_FP64, (16, 16, 48)), ((48, 48, 48), MC, m.MHD_FP64, (16, 16, 3)),
    ((32, 8, 11), MC, m.MHD_FP64, (16, 16, 2)), ((37, 4, 202), MC, m.MHD_FP64, (32, 8, 4)),
    ((256, 256, 256), WZ, m.MHD_FP64, (32, 8, 48)), ((65, 9, 7), WZ, m.MHD_FP64, (32, 4, 4)),
    ((512, 512, 512), MC, m.MHD_FP32, (32, 8, 96)),
    ((300, 200, 1), MC, m.MHD_FP64, (32, 8, 1)), ((300, 200, 1), WZ, m.MHD_FP32, (32, 4, 1)),
    ((1024, 1, 1), MC, m.MHD_FP64, (32, 1, 1))])
def test_plans_of_named_grids(n, limiter, prec, tile):
    p = m.mhd_plan_stage(m.Config(n=n, limiter=limiter, precision=prec).c(), 152)
    assert (p["tx"], p["ty"], p["tz"]) == tile


@pytest.mark.parametrize("n,prec,warps", [(32 * 608, m.MHD_FP32, 2), (32 * 608 + 1, m.MHD_FP32, 1),
                                          (1 << 20, m.MHD_FP32, 1), (1 << 20, m.MHD_FP64, 2)])
@pytest.mark.parametrize("limiter", [MC, WZ])
def test_warps_of_1d_tiles(n, prec, warps, limiter):
    assert m.mhd_plan_stage(m.Config(n=(n, 1, 1), limiter=limiter, precision=prec).c(),
                            152)["warps"] == warps


def test_bad_arguments_are_rejected():
    ok = m.Config(n=(8, 8, 8)).c()
    for cfg, nsm in [(ok, 0), (m.Config(n=(8, 1, 8)).c(), 152),
                     (m.Config(n=(8, 8, 8), rk_order=4).c(), 152)]:
        with pytest.raises(m.MHDError):
            m.mhd_plan_stage(cfg, nsm)
    assert m.lib().mhd_plan_stage(None, 152, None, None) == m.MHD_ERR_INVALID

"""The FP64 throughput probe measures the unit's full rate, that of fused
multiply-adds on register operands.  One warp issues one every 64 clocks in any
form, the full unit one every 16 (nominal 2 lanes/clk/SM) on register operands and
one every 19.1 with a constant operand: the ratio of the two rates, in which
the clock cancels, is 4.0 or 3.35; the bound lies halfway."""
import pytest

pytestmark = pytest.mark.gpu


def test_probe_reaches_the_register_operand_rate():
    import paper_2510_24175_gb300 as m
    one, full = (m.mhd_fp64_fma_rate(mask)["lane_fma_per_s"] for mask in (0x1, 0xFF))
    assert full >= 3.68 * one

"""gdws_plan_form: the library takes the folded form where its estimate is lower, and never against an option."""
import time

import numpy as np
import pytest

from paper_2110_14871_b200 import build as gbuild
from paper_2110_14871_b200 import gdws


@pytest.fixture(scope="module", autouse=True)
def built():
    gbuild.build_library()


def _plan(C, D, k, stride, g, dw_math=0):
    plan = gdws.Plan(C, D, k, stride, k // 2, np.full(C, g, dtype=np.int32))
    plan.set_option(gdws.OPT_DW_MATH, dw_math)
    return plan


@pytest.mark.parametrize("C,D,k,stride,g,n,h,form", [
    (64, 64, 3, 1, 5, 512, 32, 3),         # C k^2 D is close to G (k^2 + D): one convolution at full tensor-core rate
    (512, 512, 3, 1, 2, 32, 28, 1),        # few filters per channel in a wide layer: two stages take a quarter of the products
    (64, 64, 3, 3, 5, 8, 32, 1),           # stride 3: not covered by the folded kernel
    (60, 64, 3, 1, 5, 8, 32, 1),           # C not a multiple of 8
])
def test_form_follows_the_estimates(C, D, k, stride, g, n, h, form):
    plan = _plan(C, D, k, stride, g)
    assert plan.form(n, h, h) == form
    plan.destroy()


@pytest.mark.parametrize("dw_math", [1, 2, 3])
def test_option_overrides_the_estimates(dw_math):
    plan = _plan(64, 64, 3, 1, 5, dw_math)
    assert plan.form(512, 32, 32) == dw_math
    with pytest.raises(gdws.GdwsError):
        plan.form(0, 32, 32)
    plan.destroy()


def test_unused_channels_keep_the_two_stages():
    """g_c = 0: the folded form would multiply the channel by zero filters."""
    g = np.full(64, 5, dtype=np.int32)
    g[63] = 0
    plan = gdws.Plan(64, 64, 3, 1, 1, g)
    assert plan.form(512, 32, 32) == plan.gdw_stage() == 2
    plan.destroy()


@pytest.mark.parametrize("H,W", [(1, 9), (9, 1), (1, 1)])
@pytest.mark.parametrize("g", [2, 6])
def test_stride_2_on_one_row_or_column_is_the_alu_kernel(g, H, W):
    """The kernels that read one view per parity refuse an input without odd rows or columns."""
    plan = _plan(64, 64, 3, 2, g)
    assert plan.form(4, H, W) == 1 and plan.form(64, 64, 64) != 1
    plan.destroy()


def test_gdw_stage_is_one_of_the_two_stages():
    for g, stage in ((2, 1), (6, 2)):
        plan = _plan(64, 64, 3, 1, g, 3)
        assert plan.gdw_stage() == stage and plan.form(4, 9, 9) == 3
        plan.destroy()


@pytest.mark.parametrize("C,D,k,g,n,h", [(384, 104, 3, 2, 1, 8), (120, 256, 5, 2, 13, 5), (432, 344, 3, 2, 1, 5)])
def test_small_maps_with_stride_2_keep_the_alu_kernel(C, D, k, g, n, h):
    """A tile with few pixels costs the ALU kernel little, the folded one on pairs of SMs its full products: 1.3 to 1.7 times the time.  (In
    slices the first layer would take 7.3 us instead of 12.5; the choice counts them above two filters per channel only.)"""
    plan = _plan(C, D, k, 2, g)
    assert plan.form(n, h, h) == 1
    plan.destroy()


def test_kernel_agrees_with_form():
    """gdws_plan_kernel: form 3 is the pairs' kernel or the slices', the others their own."""
    for C, D, k, stride, g, n, h, kernel in [(64, 64, 3, 1, 5, 512, 32, gdws.KERNEL_FOLDED_PAIRS), (256, 256, 3, 1, 3, 1, 14, gdws.KERNEL_FOLDED_SLICES),
                                             (512, 512, 3, 1, 2, 32, 28, gdws.KERNEL_TWO_STAGES_ALU)]:
        plan = _plan(C, D, k, stride, g)
        assert plan.kernel(n, h, h) == kernel and min(plan.kernel(n, h, h), 3) == plan.form(n, h, h)
        plan.destroy()
    plan = _plan(64, 64, 3, 1, 5)
    assert plan.kernel(64, 28, 28, gdws.F32) == gdws.KERNEL_F32_PIECES and plan.kernel(64, 56, 56, stage=True) == gdws.KERNEL_GDW_TC
    plan.set_option(gdws.OPT_DW_MATH, 1)
    assert plan.kernel(64, 28, 28, gdws.F32) == gdws.KERNEL_F32_ALU and plan.kernel(64, 56, 56, stage=True) == gdws.KERNEL_GDW_ALU
    for bad in [lambda: plan.kernel(0, 28, 28), lambda: plan.kernel(1, 28, 28, 7), lambda: plan.kernel(1, 28, 28, gdws.F32, stage=True)]:
        with pytest.raises(gdws.GdwsError):
            bad()
    plan.destroy()


@pytest.mark.parametrize("k", [3, 5])
def test_fp32_with_few_intermediate_channels_stays_on_the_alus(k):
    """Below 16 of them the products in pieces are less exact than fp32 sums."""
    for G, kernel in [(1, gdws.KERNEL_F32_ALU), (8, gdws.KERNEL_F32_ALU), (15, gdws.KERNEL_F32_ALU), (16, gdws.KERNEL_F32_PIECES), (64, gdws.KERNEL_F32_PIECES)]:
        plan = _plan(G, 64, k, 1, 1)
        assert plan.kernel(39, 145, 145, gdws.F32) == kernel
        plan.destroy()


def test_a_first_call_on_a_large_map_takes_no_longer_to_plan():
    """The fp32 tile is looked for once per size: the search does not go through every height and width of a large map."""
    def least_us(h):
        us = []
        for _ in range(30):
            plan = _plan(64, 64, 3, 1, 5)
            t0 = time.perf_counter()
            plan.kernel(2, h, h, gdws.F32)
            us.append(1e6 * (time.perf_counter() - t0))
            plan.destroy()
        return min(us)

    assert least_us(500) <= 10 * least_us(28)        # it was 100 times


def _clusters_decide():
    """Layers that slices would take if more clusters ran at a time than do on a B200 (74, 45, 33, 26, 22, 15, 15 of 2 to 8 blocks)."""
    for N, C, D, H, k, stride, G in [(5, 32, 32, 19, 5, 1, 72), (6, 136, 272, 12, 5, 1, 649), (2, 72, 216, 17, 5, 1, 175), (54, 88, 184, 5, 5, 1, 220)]:
        g = np.full(C, G // C, dtype=np.int32)
        g[:G % C] += 1
        plan = gdws.Plan(C, D, k, stride, k // 2, g)
        got = plan.kernel(N, H, H)
        plan.destroy()
        yield got


def test_a_host_without_a_gpu_answers_as_a_b200():
    assert list(_clusters_decide()) == [gdws.KERNEL_FOLDED_PAIRS] * 4


@pytest.mark.gpu
def test_a_b200_answers_as_a_host_without_a_gpu():
    assert list(_clusters_decide()) == [gdws.KERNEL_FOLDED_PAIRS] * 4

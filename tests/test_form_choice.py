"""gdws_plan_form: the library takes the folded form where its estimate is lower, and never against an option."""
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

"""Folded filters formed when weights are packed: windows whose filters need several stages of shared memory, filters that start and end
off the wide loads' boundaries, channels without filters, output channels off the blocks of four, weights in bf16 and fp32; and the time
that it adds to a call given its weights."""
import numpy as np
import pytest
import torch

from paper_2110_14871_b200 import build as gbuild
from paper_2110_14871_b200 import gdws
from paper_2110_14871_b200 import inputs as gi

from util import make_plan, rel_err, run_oracle, small_spec, to_device

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    gbuild.build_library()


@pytest.mark.parametrize("N,C,D,H,W,k,gd", [
    (1, 8, 8, 5, 5, 3, ("const", 1)),                  # 72 taps: less than a load per thread
    (2, 72, 40, 9, 7, 3, ("uniform", 0, 9)),           # a second window of 8 channels that starts anywhere
    (1, 64, 24, 8, 8, 3, ("const", 25)),               # 1600 filters of 9 taps: two stages (942 fit)
    (1, 72, 16, 6, 6, 5, ("uniform", 7, 25)),          # 25 taps: three (422 fit)
    (1, 16, 32, 7, 7, 5, ("const", 70)),
    (2, 24, 136, 6, 9, 4, ("uniform", 1, 16)),
    (1, 8, 264, 5, 5, 2, ("uniform", 1, 3)),
    (1, 512, 264, 5, 5, 3, ("uniform", 1, 3)),         # four output channels per thread
])
def test_folded_filters_match_reference(N, C, D, H, W, k, gd):
    data = gi.make_layer(small_spec("t", N, C, D, H, W, k, 1, k // 2, gd, "bf16", "NHWC", seed=C + D + k))
    plan = make_plan(data, path=gdws.PATH_FUSED, dw_math=3)
    x, b = to_device(data.x, "bf16"), torch.from_numpy(data.bias).cuda()
    ys = []
    for dtype in ("bf16", "f32"):                      # the same values
        y = torch.full((N, data.spec.Ho, data.spec.Wo, D), float("nan"), dtype=torch.bfloat16, device="cuda")
        plan.pack_weights(to_device(data.dw_w, dtype), to_device(data.pw_w, dtype), b)
        plan.forward(x, y, "NHWC")
        ys.append(y)
    torch.cuda.synchronize()
    plan.status()
    assert torch.equal(ys[0], ys[1])
    assert rel_err(ys[0].float().cpu().numpy(), run_oracle(data)[0]) <= 1e-2      # folded filters and y rounded once each, and sums
    plan.destroy()


@pytest.mark.parametrize("N,C,D,H,k,gd,most", [(4, 56, 40, 6, 5, ("heavy",), 2.5), (8, 48, 64, 34, 5, ("uniform", 1, 25), 5.0), (2, 72, 120, 13, 3, ("uniform", 1, 9), 2.5)])
def test_folding_adds_little_to_a_call_given_its_weights(N, C, D, H, k, gd, most):
    """What packing takes in front of a folded forward against what it takes in front of the two stages, which is part of the same launch:
    2.3 times at most, 3.4 with up to 25 filters a channel (2.7 and 7.6 when each thread fetched its own filters)."""
    data = gi.make_layer(small_spec("t", N, C, D, H, H, k, 1, k // 2, gd, "bf16", "NHWC", seed=3))
    plan = make_plan(data, path=gdws.PATH_FUSED)
    x, dw, pw, b = to_device(data.x, "bf16"), to_device(data.dw_w, "bf16"), to_device(data.pw_w, "bf16"), torch.from_numpy(data.bias).cuda()
    y = torch.empty((N, H, H, D), dtype=torch.bfloat16, device="cuda")

    def least_us(w):
        graph = torch.cuda.CUDAGraph()
        plan.forward(x, y, "NHWC", *w)
        torch.cuda.synchronize()
        with torch.cuda.graph(graph):
            for _ in range(20):
                plan.forward(x, y, "NHWC", *w)
        us = []
        for _ in range(6):
            a, e = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            graph.replay()
            e.record()
            torch.cuda.synchronize()
            us.append(a.elapsed_time(e) * 50)
        return min(us)

    extra = {}
    for m in (1, 3):
        plan.set_option(gdws.OPT_DW_MATH, m)
        extra[m] = least_us((dw, pw, b))
        plan.pack_weights(dw, pw, b)
        extra[m] -= least_us(())
    plan.status()
    plan.destroy()
    assert extra[3] <= most * extra[1], extra

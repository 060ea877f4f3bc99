"""The folded form on pairs of SMs, in batches large enough that it runs there: both strides, filter sizes of one to five, maps at most
4 wide (a load per tap), short last windows, output channels just past 256, filters with and without their second term."""
import numpy as np
import pytest
import torch

from oracle import gdws_oracle as orc
from paper_2110_14871_b200 import build as gbuild
from paper_2110_14871_b200 import gdws
from paper_2110_14871_b200 import inputs as gi

from util import Guarded, make_plan, rel_err, small_spec, to_device

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    gbuild.build_library()


@pytest.mark.parametrize("zero_sum", [False, True])
@pytest.mark.parametrize("N,C,D,H,W,k,stride,pad", [
    (140, 24, 40, 20, 17, 3, 2, 1), (320, 64, 96, 16, 16, 3, 2, 1), (1290, 72, 64, 8, 8, 3, 2, 1), (610, 136, 72, 4, 4, 3, 1, 1),
    (1290, 16, 128, 3, 3, 3, 1, 1), (12, 72, 120, 20, 19, 3, 1, 1), (21, 80, 264, 14, 14, 3, 1, 1), (40, 24, 40, 19, 23, 5, 2, 2),
    (110, 16, 32, 12, 12, 4, 1, 1), (110, 16, 8, 12, 10, 2, 1, 0), (380, 40, 24, 7, 7, 1, 1, 0), (420, 16, 16, 12, 12, 1, 2, 0),
    (260, 136, 264, 6, 5, 3, 1, 0), (160, 128, 96, 17, 19, 3, 2, 0), (80, 64, 64, 20, 20, 5, 1, 0), (53, 520, 520, 7, 7, 3, 1, 0),
    (1290, 16, 24, 4, 4, 5, 1, 2), (810, 24, 32, 9, 4, 3, 2, 1),
])
def test_pairs_match_reference(N, C, D, H, W, k, stride, pad, zero_sum):
    data = gi.make_layer(small_spec("t", N, C, D, H, W, k, stride, pad, ("const", 3), "bf16", "NHWC", relu=C == 72, seed=C + D + k))
    s = data.spec
    if zero_sum and k > 1:
        data.dw_w[...] = torch.from_numpy(data.dw_w - data.dw_w.mean(axis=(1, 2), keepdims=True)).to(torch.bfloat16).float().numpy()
    plan = make_plan(data, path=gdws.PATH_FUSED, dw_math=3)
    assert plan.kernel(N, H, W) == gdws.KERNEL_FOLDED_PAIRS
    plan.pack_weights(to_device(data.dw_w, "bf16"), to_device(data.pw_w, "bf16"), torch.from_numpy(data.bias).cuda())
    x = to_device(data.x, "bf16")
    yg = Guarded((N, s.Ho, s.Wo, D), torch.bfloat16)
    got = []
    for _ in range(2):
        yg.t.fill_(float("nan"))
        plan.forward(x, yg.t, "NHWC")
        torch.cuda.synchronize()
        plan.status()
        got.append(yg.t.float().cpu().numpy())
    yg.check("y")
    assert np.array_equal(got[0], got[1])
    some = sorted({0, 1, N // 3, N // 2, N - 2, N - 1})                  # images are independent
    ref, _ = orc.forward(data.x[some], data.g, data.dw_w, data.pw_w, data.bias, stride=stride, pad=pad, relu=s.relu, layout="NHWC")
    assert rel_err(got[0][some], ref) <= 1e-2        # folded filters and y rounded once each: 2^-8 and 2^-9, and sums
    plan.destroy()

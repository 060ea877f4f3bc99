"""The folded form in slices: small layers whose sum over channels and filter rows is shared by the blocks of a cluster.  Several
slices and one, tiles of several images, maps at most 4 wide, both strides and filter sizes, a last window of few channels, output
channels off the blocks of 32, fp32 output, ReLU, and filters that take their second term."""
import numpy as np
import pytest
import torch

from paper_2110_14871_b200 import build as gbuild
from paper_2110_14871_b200 import gdws
from paper_2110_14871_b200 import inputs as gi

from util import Guarded, make_plan, rel_err, run_oracle, small_spec, to_device

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    gbuild.build_library()


@pytest.mark.parametrize("zero_sum", [False, True])
@pytest.mark.parametrize("N,C,D,H,W,k,stride", [
    (1, 256, 256, 14, 14, 3, 1), (1, 512, 504, 7, 7, 3, 1), (4, 448, 264, 4, 4, 3, 1), (3, 72, 120, 20, 20, 3, 1), (5, 136, 200, 6, 5, 3, 1),
    (9, 128, 64, 16, 16, 5, 2), (2, 200, 8, 9, 11, 3, 2), (1, 24, 40, 16, 16, 3, 1), (2, 328, 40, 3, 9, 5, 1),
])
def test_slices_match_reference(N, C, D, H, W, k, stride, zero_sum):
    data = gi.make_layer(small_spec("t", N, C, D, H, W, k, stride, k // 2, ("uniform", 3, 5), "bf16", "NHWC", relu=N == 3, seed=C + D))
    s, f32 = data.spec, N in (1, 5)
    if zero_sum:
        data.dw_w[...] = torch.from_numpy(data.dw_w - data.dw_w.mean(axis=(1, 2), keepdims=True)).to(torch.bfloat16).float().numpy()
    plan = make_plan(data)
    plan.set_option(gdws.OPT_OUT_DTYPE, int(f32))
    assert plan.form(N, H, W) == 3 and plan.kernel(N, H, W) == gdws.KERNEL_FOLDED_SLICES
    plan.pack_weights(to_device(data.dw_w, "bf16"), to_device(data.pw_w, "bf16"), torch.from_numpy(data.bias).cuda())
    x = to_device(data.x, "bf16")
    yg = Guarded((N, s.Ho, s.Wo, D), torch.float32 if f32 else torch.bfloat16)
    got = []
    for _ in range(2):
        yg.t.fill_(float("nan"))
        plan.forward(x, yg.t, "NHWC")
        torch.cuda.synchronize()
        plan.status()
        got.append(yg.t.float().cpu().numpy())
    yg.check("y")
    assert np.array_equal(got[0], got[1])
    assert rel_err(got[0], run_oracle(data)[0]) <= 1e-2        # folded filters and y rounded once each: 2^-8 and 2^-9, and sums
    plan.destroy()


@pytest.mark.parametrize("N,D", [(2, 264), (4, 264)])
def test_every_cluster_of_three_right_after_packing(N, D):
    """A layer that takes all of the clusters of three that fit, given its weights: no more than packing, then the forward, and a launch
    between them (its last clusters came in a second round when the launches overlapped: 5 to 8 us more)."""
    data = gi.make_layer(small_spec("t", N, 448, D, 20, 20, 3, 1, 1, ("uniform", 1, 5), "bf16", "NHWC", seed=3))
    plan = make_plan(data)
    assert plan.kernel(N, 20, 20) == gdws.KERNEL_FOLDED_SLICES
    x, dw, pw, b = to_device(data.x, "bf16"), to_device(data.dw_w, "bf16"), to_device(data.pw_w, "bf16"), torch.from_numpy(data.bias).cuda()
    y = torch.empty((N, 20, 20, D), dtype=torch.bfloat16, device="cuda")

    def least_us(call):
        call()
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            for _ in range(20):
                call()
        us = []
        for _ in range(6):
            a, e = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            graph.replay()
            e.record()
            torch.cuda.synchronize()
            us.append(a.elapsed_time(e) * 50)
        return min(us)

    given = least_us(lambda: plan.forward(x, y, "NHWC", dw, pw, b))
    pack = least_us(lambda: plan.pack_weights(dw, pw, b))
    packed = least_us(lambda: plan.forward(x, y, "NHWC"))
    plan.status()
    plan.destroy()
    assert given <= pack + packed + 3.0, (given, pack, packed)

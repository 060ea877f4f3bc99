"""Precision of the folded form.  Its filters are rounded to bf16 where the two-stage kernels round z; filters that cut a constant
input off (their taps sum to zero) are taken in two bf16 terms, because one term's rounding errors would add up on the input's
mean.  Errors are 2-norms relative to the fp64 reference; rounding y to nearest alone is at most 2^-8 / sqrt(3) of it."""
import numpy as np
import pytest
import torch

from paper_2110_14871_b200 import build as gbuild
from paper_2110_14871_b200 import gdws
from paper_2110_14871_b200 import inputs as gi

from util import make_plan, run_gpu, run_oracle, small_spec, to_device

pytestmark = pytest.mark.gpu

ROUND_Y = 2.0 ** -8 / 3 ** 0.5


@pytest.fixture(scope="module", autouse=True)
def built():
    gbuild.build_library()


def _err(y, ref):
    return float(np.linalg.norm(y - ref) / np.linalg.norm(ref))


def _zero_sums(dw):
    """Taps that are multiples of 1/32 (exact in bf16) and sum to zero."""
    q = np.round(dw * 16)
    c = q.shape[1] // 2
    q[:, c, c] -= q.sum((1, 2))
    return (q / 32).astype(np.float32)


SHAPES = [
    # N, C, D, H, W, k, stride, g_dist
    (3, 64, 64, 21, 18, 3, 1, ("uniform", 3, 7)),       # one window and box: two issuing threads with one term
    (150, 64, 64, 18, 18, 3, 1, ("uniform", 3, 7)),     # several items per pair; filters that would stay
    (2, 72, 120, 20, 19, 3, 1, ("uniform", 1, 9)),      # a second window of 8 channels
    (40, 256, 256, 20, 20, 3, 1, ("uniform", 1, 3)),    # ring of filters
    (6, 128, 96, 17, 19, 3, 2, ("uniform", 1, 9)),      # four views, two loads per box
    (4, 136, 264, 6, 5, 3, 1, ("uniform", 1, 9)),       # maps at most 4 wide, two blocks of output channels
    (3, 64, 64, 20, 20, 5, 1, ("uniform", 3, 12)),      # 25 taps: a sum runs over all of them
    (2, 24, 40, 19, 23, 5, 2, ("uniform", 3, 12)),
    (2, 16, 32, 16, 14, 2, 1, ("uniform", 1, 4)),
    (1, 520, 520, 7, 7, 3, 1, ("uniform", 1, 2)),       # sums from every n-th group of output channels
]


@pytest.mark.parametrize("mean", [10.0, 100.0])
@pytest.mark.parametrize("shape", SHAPES)
def test_zero_sum_filters_on_inputs_with_a_mean(shape, mean):
    N, C, D, H, W, k, stride, gd = shape
    data = gi.make_layer(small_spec("t", N, C, D, H, W, k, stride, 0, gd, "bf16", "NHWC", seed=61 + C + k))
    data.dw_w[...] = _zero_sums(data.dw_w)
    data.x[...] = gi.round_to_bf16(data.x + np.float32(mean))
    ref, _ = run_oracle(data)
    for dw_math in (3, 0):
        assert _err(run_gpu(data, path=gdws.PATH_FUSED, dw_math=dw_math), ref) <= (ROUND_Y if dw_math == 3 else 2 ** 0.5 * ROUND_Y)


@pytest.mark.parametrize("x", ["normal", "mean", "relu"])
@pytest.mark.parametrize("shape", SHAPES[1:8])
def test_ordinary_filters_are_as_precise_as_two_stages(shape, x):
    """sqrt(2) ROUND_Y: y's rounding and one before it.  Against each other: on inputs with a mean a part of the error is the same
    for all pixels, so its size is that of D independent values and scatters by 1 / sqrt(2 D) on either side."""
    N, C, D, H, W, k, stride, gd = shape
    data = gi.make_layer(small_spec("t", min(N, 12), C, D, H, W, k, stride, 0, gd, "bf16", "NHWC", seed=71 + C + k))
    if x != "normal":
        data.x[...] = gi.round_to_bf16(data.x + np.float32(1.0)) if x == "mean" else np.maximum(data.x, 0)
    ref, _ = run_oracle(data)
    err = {m: _err(run_gpu(data, path=gdws.PATH_FUSED, dw_math=m), ref) for m in (1, 3)}
    assert err[3] <= (1.05 if x == "normal" else 1 + 2 / D ** 0.5) * err[1] and err[3] <= 2 ** 0.5 * ROUND_Y, err


def test_weights_of_both_kinds_in_turn():
    """One plan, packed with ordinary and with zero-sum filters alternately: each forward is bit for bit that of a plan of its own."""
    data = gi.make_layer(small_spec("t", 90, 64, 96, 16, 16, 3, 1, 1, ("uniform", 3, 7), "bf16", "NHWC", seed=83))
    data.x[...] = gi.round_to_bf16(data.x + np.float32(10.0))
    pw, b, x = to_device(data.pw_w, "bf16"), torch.from_numpy(data.bias).cuda(), to_device(data.x, "bf16")
    kinds = [to_device(data.dw_w, "bf16"), to_device(_zero_sums(data.dw_w), "bf16")]
    s = data.spec

    def forward(plan, dw):
        y = torch.full((s.N, s.Ho, s.Wo, s.D), float("nan"), dtype=torch.bfloat16, device="cuda")
        plan.forward(x, y, "NHWC", dw, pw, b)
        return y

    own = []
    for dw in kinds:
        plan = make_plan(data, path=gdws.PATH_FUSED, dw_math=3)
        own.append(forward(plan, dw))
        torch.cuda.synchronize()
        plan.destroy()
    plan = make_plan(data, path=gdws.PATH_FUSED, dw_math=3)
    got = [forward(plan, kinds[i % 2]) for i in range(6)]
    torch.cuda.synchronize()
    plan.status()
    assert all(torch.equal(g, own[i % 2]) for i, g in enumerate(got))
    plan.destroy()

"""The folded form of the bf16 forward (one k x k convolution with filters formed at pack time) against the CPU reference.
The reference takes the two stages in fp64; the kernel rounds each folded filter tap to bf16 once (relative error up to
2^-8) where the two-stage kernels round z, and both round y: the bound of the other bf16 kernels, 1e-2, applies."""
import numpy as np
import pytest
import torch

from paper_2110_14871_b200 import build as gbuild
from paper_2110_14871_b200 import gdws
from paper_2110_14871_b200 import inputs as gi

from util import Guarded, make_plan, rel_err, run_gpu, run_oracle, small_spec, to_device

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    gbuild.build_library()


SHAPES = [
    # N, C, D, H, W, k, stride, pad, g_dist
    (1, 64, 64, 16, 16, 3, 1, 1, ("uniform", 1, 9)),        # one pair of whole tiles
    (1, 8, 8, 5, 5, 3, 1, 1, ("uniform", 0, 9)),            # smallest channels: one K step, a quarter of a staged block
    (3, 72, 120, 45, 19, 3, 1, 1, ("heavy",)),              # ragged map, second window of 8 channels, odd number of tiles
    (2, 80, 264, 14, 14, 3, 1, 1, ("heavy",)),              # D beyond 256: two blocks of output channels
    (5, 128, 128, 8, 8, 3, 1, 1, ("uniform", 1, 9)),        # two images per tile
    (9, 136, 72, 4, 4, 3, 1, 1, ("uniform", 1, 9)),         # 4-wide maps: one copy per tap
    (4, 16, 128, 3, 3, 3, 1, 1, ("uniform", 1, 9)),
    (150, 64, 64, 16, 16, 3, 1, 1, ("uniform", 1, 9)),      # more work items than pairs of SMs: both accumulators, filters resident
    (40, 256, 256, 28, 20, 3, 1, 1, ("heavy",)),            # the same with the filter ring
    (2, 192, 512, 10, 9, 3, 1, 1, ("uniform", 1, 3)),
    (2, 24, 40, 20, 17, 3, 2, 1, ("uniform", 1, 9)),        # stride 2: four views, odd sizes
    (6, 64, 96, 16, 16, 3, 2, 1, ("uniform", 1, 9)),        # 8 x 8 outputs
    (9, 72, 64, 8, 8, 3, 2, 1, ("uniform", 1, 9)),          # 4 x 4 outputs
    (2, 16, 24, 13, 11, 5, 1, 2, ("uniform", 1, 25)),
    (30, 96, 160, 30, 30, 5, 1, 2, ("heavy",)),
    (2, 24, 40, 19, 23, 5, 2, 2, ("uniform", 1, 25)),
    (2, 16, 32, 12, 12, 4, 1, 1, ("uniform", 1, 16)),
    (1, 16, 8, 12, 10, 2, 1, 0, ("uniform", 1, 4)),
    (2, 40, 24, 7, 7, 1, 1, 0, ("uniform", 1, 1)),
    (2, 16, 16, 12, 12, 1, 2, 0, ("uniform", 1, 1)),
]


@pytest.mark.parametrize("shape", SHAPES)
def test_folded_forward_matches_reference(shape):
    N, C, D, H, W, k, s, p, gd = shape
    spec = small_spec("t", N, C, D, H, W, k, s, p, gd, "bf16", "NHWC", relu=(C % 16 == 8), seed=11 + sum(shape[:8]))
    data = gi.make_layer(spec)
    y = run_gpu(data, path=gdws.PATH_FUSED, dw_math=3, prepack=C > 64)
    ref, _ = run_oracle(data)
    assert rel_err(y, ref) <= 1e-2


@pytest.mark.parametrize("shape", [(3, 32, 40, 12, 9), (2, 64, 264, 20, 20), (150, 16, 48, 16, 16)])
def test_folded_fp32_output_rounds_to_the_bf16_output(shape):
    N, C, D, H, W = shape
    spec = small_spec("t", N, C, D, H, W, 3, 1, 1, ("uniform", 1, 9), "bf16", "NHWC", relu=True, seed=91)
    data = gi.make_layer(spec)
    want16 = run_gpu(data, path=gdws.PATH_FUSED, dw_math=3)
    plan = make_plan(data, path=gdws.PATH_FUSED, dw_math=3)
    plan.set_option(gdws.OPT_OUT_DTYPE, 1)
    x, dw, pw = (to_device(a, "bf16") for a in (data.x, data.dw_w, data.pw_w))
    yg = Guarded((spec.N, spec.Ho, spec.Wo, spec.D), torch.float32, fill=float("nan"))
    plan.forward(x, yg.t, "NHWC", dw, pw, torch.from_numpy(data.bias).cuda())
    torch.cuda.synchronize()
    plan.status()
    yg.check("y")
    assert np.array_equal(yg.t.to(torch.bfloat16).float().cpu().numpy().astype(np.float64), want16)
    plan.destroy()


def test_folded_refuses_what_it_does_not_cover():
    data = gi.make_layer(small_spec("t", 2, 16, 16, 9, 9, 3, 3, 1, seed=78))
    with pytest.raises(gdws.GdwsError) as e:
        run_gpu(data, path=gdws.PATH_FUSED, dw_math=3)
    assert e.value.status == gdws.ERR_UNSUPPORTED


def test_folded_filters_keep_their_sums_on_inputs_with_a_mean():
    """Inputs of mean 4 and unit spread, ordinary filters: what their taps' rounding adds on the mean is no more than what
    rounding z adds in the two-stage kernels.  Both are compared with the reference in the 2-norm, where y's own rounding
    (up to 2^-8 / sqrt(3) of each value) dominates."""
    spec = small_spec("t", 3, 64, 64, 20, 20, 3, 1, 0, ("uniform", 3, 7), "bf16", "NHWC", seed=53)
    data = gi.make_layer(spec)
    data.x = gi.round_to_bf16(data.x + 4.0)
    ref, _ = run_oracle(data)
    err = {m: float(np.linalg.norm(run_gpu(data, path=gdws.PATH_FUSED, dw_math=m) - ref) / np.linalg.norm(ref)) for m in (1, 3)}
    assert err[3] <= 1.1 * err[1], err

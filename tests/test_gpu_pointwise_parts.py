"""gdws_pointwise with an item's output channels cut: more than 256 of them, and few pixels (down to 64 channels an item), the last part
narrower than the others, channels off the multiples of 16, fp32 output."""
import numpy as np
import pytest
import torch

from paper_2110_14871_b200 import build as gbuild
from paper_2110_14871_b200 import gdws
from paper_2110_14871_b200 import inputs as gi

from util import Guarded, make_plan, rel_err, small_spec, to_device

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    gbuild.build_library()


@pytest.mark.parametrize("f32", [False, True])
@pytest.mark.parametrize("N,C,D,H,W", [(1, 24, 264, 5, 5), (2, 40, 416, 8, 5), (1, 16, 512, 13, 11), (3, 8, 136, 9, 9), (2, 72, 200, 1, 1), (40, 16, 392, 24, 23), (40, 24, 72, 24, 23)])
def test_parts_of_the_output_channels(N, C, D, H, W, f32):
    data = gi.make_layer(small_spec("t", N, C, D, H, W, 3, 1, 1, ("uniform", 1, 5), "bf16", "NHWC", relu=N == 2, seed=C + D))
    plan = make_plan(data)
    plan.set_option(gdws.OPT_OUT_DTYPE, int(f32))
    plan.pack_weights(to_device(data.dw_w, "bf16"), to_device(data.pw_w, "bf16"), torch.from_numpy(data.bias).cuda())
    G, Gp, _, _ = plan.info()
    z = torch.randn((N * H * W, Gp), generator=torch.Generator(device="cuda").manual_seed(D), device="cuda").to(torch.bfloat16)
    z[:, G:] = 0
    yg = Guarded((N, H, W, D), torch.float32 if f32 else torch.bfloat16, fill=float("nan"))
    plan.pointwise(z, yg.t, "NHWC")
    torch.cuda.synchronize()
    plan.status()
    yg.check("y")
    want = z[:, :G].cpu().double().numpy() @ data.pw_w.astype(np.float64).T + data.bias
    want = (np.maximum(want, 0) if data.spec.relu else want).reshape(N, H, W, D)
    assert rel_err(yg.t.float().cpu().numpy(), want) <= (1e-5 if f32 else 2 ** -8)      # sums of up to 400 exact products; y rounded once
    plan.destroy()

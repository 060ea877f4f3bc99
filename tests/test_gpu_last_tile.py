"""Two-stage kernel with few chunks per tile and several tiles per block: the depthwise warps run tiles ahead of the tensor
cores, and the ones that help with a block's last tile must wait for that tile's sums, not for an earlier tile's.  (Outputs
beyond 256 channels, fp32 outputs and D off the multiples of 64 are stored by those warps too.)"""
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


@pytest.mark.parametrize("N,C,D,H,W,k,g,out_f32", [
    (8, 16, 480, 60, 76, 5, 4, True),        # one chunk per tile, one accumulator
    (8, 16, 480, 60, 76, 5, 4, False),
    (12, 16, 368, 48, 48, 3, 8, False),       # two chunks
    (14, 32, 512, 48, 40, 5, 5, True),        # three chunks
    (8, 32, 272, 56, 56, 3, 8, False),       # four chunks
    (12, 64, 200, 56, 56, 3, 1, False),      # one chunk, two accumulators
    (12, 64, 256, 56, 56, 3, 1, True),
    (5, 16, 480, 60, 76, 2, 4, False),       # generic depthwise code
])
def test_last_tile_of_a_block(N, C, D, H, W, k, g, out_f32):
    data = gi.make_layer(small_spec("t", N, C, D, H, W, k, 1, k // 2, ("const", g), "bf16", "NHWC", seed=N + C + D + k))
    s = data.spec
    ref, _ = run_oracle(data)
    plan = make_plan(data, path=gdws.PATH_FUSED, dw_math=1)
    plan.set_option(gdws.OPT_OUT_DTYPE, int(out_f32))
    assert plan.tile(N, H, W)[3] > 148       # a block has a second tile
    plan.pack_weights(to_device(data.dw_w, "bf16"), to_device(data.pw_w, "bf16"), torch.from_numpy(data.bias).cuda())
    x = to_device(data.x, "bf16")
    yg = Guarded((s.N, s.Ho, s.Wo, s.D), torch.float32 if out_f32 else torch.bfloat16)
    first = None
    for _ in range(3):
        yg.t.fill_(float("nan"))
        plan.forward(x, yg.t, "NHWC")
        torch.cuda.synchronize()
        plan.status()
        y = yg.t.float().cpu().numpy().astype(np.float64)
        assert rel_err(y, ref) <= 1e-2       # z and y rounded to bf16
        assert first is None or np.array_equal(first, y)
        first = y
    yg.check("y")
    plan.destroy()

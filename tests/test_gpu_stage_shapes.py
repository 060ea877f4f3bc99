"""gdws_depthwise where no specialised depthwise code applies (its z goes through operand stages) and where one does (z from
registers): every filter size and stride, ragged maps, several chunks and tiles per block, against the CPU reference, and bit
for bit twice."""
import numpy as np
import pytest
import torch

from paper_2110_14871_b200 import build as gbuild
from paper_2110_14871_b200 import inputs as gi

from util import Guarded, make_plan, rel_err, run_oracle, small_spec, to_device

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    gbuild.build_library()


@pytest.mark.parametrize("N,C,H,W,k,stride,g", [
    (37, 192, 7, 5, 1, 2, 3), (3, 24, 20, 17, 2, 1, 2), (2, 40, 21, 18, 3, 3, 5), (2, 16, 30, 23, 4, 1, 9), (1, 8, 25, 26, 5, 3, 7),
    (1, 8, 19, 21, 6, 2, 8), (2, 16, 33, 20, 7, 1, 5), (9, 64, 40, 40, 1, 1, 1), (40, 72, 24, 20, 1, 1, 2),
    (3, 24, 20, 17, 3, 1, 9), (9, 16, 4, 4, 3, 1, 5), (9, 16, 8, 7, 3, 2, 3), (2, 16, 20, 30, 5, 2, 9), (64, 64, 28, 28, 3, 1, 3),
])
def test_depthwise_stage(N, C, H, W, k, stride, g):
    data = gi.make_layer(small_spec("t", N, C, 16, H, W, k, stride, k // 2, ("uniform", 1, g), "bf16", "NHWC", seed=7 * k + C))
    s = data.spec
    plan = make_plan(data)
    plan.pack_weights(to_device(data.dw_w, "bf16"), to_device(data.pw_w, "bf16"))
    G, Gp, _, _ = plan.info()
    x = to_device(data.x, "bf16")
    zg = Guarded((s.N * s.Ho * s.Wo, Gp), torch.bfloat16)
    got = []
    for _ in range(2):
        zg.t.fill_(float("nan"))
        plan.depthwise(x, zg.t, "NHWC")
        torch.cuda.synchronize()
        plan.status()
        got.append(zg.t.float().cpu().numpy())
    zg.check("z")
    assert np.array_equal(got[0], got[1]) and (got[0][:, G:] == 0).all()
    _, zr, _ = run_oracle(data, return_z=True)
    assert rel_err(got[0][:, :G].reshape(s.N, s.Ho, s.Wo, G), zr) <= 2 ** -8      # z rounded once
    plan.destroy()

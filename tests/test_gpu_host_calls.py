"""gdws_forward_host calls that are cut into pieces: images whose bytes are no multiple of 16 with even pieces."""
import pytest
import torch

from paper_2110_14871_b200 import build as gbuild
from paper_2110_14871_b200 import inputs as gi

from util import TOL, make_plan, rel_err, run_oracle, small_spec, to_device

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    gbuild.build_library()


# piece sizes 28 (14 first) and 6 (3 first) images; odd image sizes of x, of y, of both
@pytest.mark.parametrize("N,C,D,H,W", [(56, 13, 15, 71, 63), (56, 13, 16, 71, 63), (56, 16, 13, 71, 63), (12, 65, 65, 63, 61), (2, 129, 131, 63, 71)])
def test_pieces_start_on_16_byte_boundaries(N, C, D, H, W):
    data = gi.make_layer(small_spec("t", N, C, D, H, W, 3, 1, 1, ("const", 1), "f32", "NCHW", seed=23))
    ref, _ = run_oracle(data)
    plan = make_plan(data)
    x = torch.from_numpy(data.x).pin_memory()
    y = torch.full(ref.shape, float("nan")).pin_memory()
    plan.forward_host(x, y, "NCHW", to_device(data.dw_w, "f32"), to_device(data.pw_w, "f32"), torch.from_numpy(data.bias).cuda())
    assert rel_err(y.numpy(), ref) <= TOL["f32"]
    plan.destroy()

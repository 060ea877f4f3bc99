"""gdws_forward_host calls that are cut into pieces: images whose bytes are no multiple of 16 with even pieces; a
workspace that holds a piece but not the batch."""
import pytest
import torch

from paper_2110_14871_b200 import build as gbuild
from paper_2110_14871_b200 import gdws
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


def test_workspace_is_checked_against_the_whole_batch():
    data = gi.make_layer(small_spec("t", 60, 16, 16, 64, 64, 3, 1, 1, ("const", 2), "bf16", "NHWC", seed=29))
    s = data.spec
    plan = make_plan(data, path=gdws.PATH_UNFUSED)
    plan.pack_weights(to_device(data.dw_w, "bf16"), to_device(data.pw_w, "bf16"), torch.from_numpy(data.bias).cuda())
    x = torch.from_numpy(data.x).to(torch.bfloat16).pin_memory()
    y = torch.full((s.N, s.Ho, s.Wo, s.D), 3.0, dtype=torch.bfloat16).pin_memory()
    need = plan.workspace_bytes(gdws.BF16, s.N, s.H, s.W)
    ws = torch.empty(need, dtype=torch.uint8, device="cuda")
    plan.set_workspace(ws[:need - 256])
    with pytest.raises(gdws.GdwsError) as e:
        plan.forward_host(x, y, "NHWC")
    assert e.value.status == gdws.ERR_WORKSPACE and bool((y == 3.0).all())
    plan.set_workspace(ws)
    plan.forward_host(x, y, "NHWC")
    ref, _ = run_oracle(data)
    assert rel_err(y.float().numpy(), ref) <= TOL["bf16"]
    plan.destroy()

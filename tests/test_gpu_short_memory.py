"""A plan for which there is memory but not for its folded filters keeps to the two stages."""
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


def test_plan_without_room_for_folded_filters():
    data = gi.make_layer(small_spec("t", 1, 1024, 512, 6, 6, 5, 1, 2, ("const", 4), "bf16", "NHWC", seed=97))
    ref, _ = run_oracle(data)
    dw, pw, x = (to_device(a, "bf16") for a in (data.dw_w, data.pw_w, data.x))
    y = torch.empty(ref.shape, dtype=torch.bfloat16, device="cuda")

    def build_and_run(fold):
        plan = make_plan(data, path=gdws.PATH_FUSED)
        assert (plan.form(1, 6, 6) == 3) == fold
        plan.forward(x, y, "NHWC", dw, pw, torch.from_numpy(data.bias).cuda())
        torch.cuda.synchronize()
        plan.status()
        assert rel_err(y.float().cpu().numpy(), ref) <= 1e-2
        plan.set_option(gdws.OPT_DW_MATH, 1)
        plan.forward(x, y, "NHWC")            # loads the ALU kernel before the memory gets short
        torch.cuda.synchronize()
        plan.destroy()

    build_and_run(True)
    torch.cuda.empty_cache()
    room = 36 << 20                           # the folded filters take 50 MB, the rest of the plan some 10
    fill = torch.empty(torch.cuda.mem_get_info()[0] - room, dtype=torch.uint8, device="cuda")
    try:
        build_and_run(False)
    finally:
        del fill
        torch.cuda.empty_cache()

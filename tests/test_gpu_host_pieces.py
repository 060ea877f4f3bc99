"""gdws_forward_host with pinned batches large enough to go through in overlapping pieces: ragged piece sizes, images whose
bytes are no multiple of 16, two calls in a row on the same buffers, weights passed with the call."""
import numpy as np
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


@pytest.mark.parametrize("dtype,N,C,D,H,W", [("bf16", 61, 64, 64, 20, 20), ("bf16", 2, 128, 256, 80, 41), ("bf16", 90, 64, 64, 56, 54), ("f32", 53, 13, 15, 71, 63)])
def test_pieces_match_reference(dtype, N, C, D, H, W):
    layout = "NHWC" if dtype == "bf16" else "NCHW"
    spec = small_spec("t", N, C, D, H, W, 3, 1, 1, ("uniform", 1, 3), dtype, layout, seed=17)
    data = gi.make_layer(spec)
    ref, _ = run_oracle(data)
    plan = make_plan(data)
    dw, pw, b = to_device(data.dw_w, dtype), to_device(data.pw_w, dtype), torch.from_numpy(data.bias).cuda()
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    x = torch.from_numpy(data.x).to(tdt).pin_memory()
    y = torch.full(ref.shape, float("nan"), dtype=tdt).pin_memory()
    for flip in (1.0, -1.0):                     # y is linear in x up to the bias: the second call sees other values
        plan.forward_host(x if flip == 1.0 else (-x).pin_memory(), y, layout, dw, pw, b)
        bias = data.bias.reshape((1, -1, 1, 1) if layout == "NCHW" else (1, 1, 1, -1)).astype(np.float64)
        assert rel_err(y.float().numpy(), flip * (ref - bias) + bias) <= TOL[dtype]
        y.fill_(float("nan"))
    plan.status()
    plan.destroy()


def test_a_layer_that_only_the_slices_cover_goes_in_pieces():
    """More than 4096 output channels on a few small maps: a piece's time is the slices' estimate, not that of a kernel that does not run."""
    data = gi.make_layer(small_spec("t", 8, 64, 4104, 8, 8, 3, 1, 1, ("const", 3), "bf16", "NHWC", seed=19))
    plan = make_plan(data)
    plan.set_option(gdws.OPT_OUT_DTYPE, 1)
    assert plan.kernel(8, 8, 8) == gdws.KERNEL_FOLDED_SLICES
    plan.pack_weights(to_device(data.dw_w, "bf16"), to_device(data.pw_w, "bf16"), torch.from_numpy(data.bias).cuda())
    x = torch.from_numpy(data.x).to(torch.bfloat16).pin_memory()
    ref, _ = run_oracle(data)
    y = torch.full(ref.shape, float("nan")).pin_memory()
    before = plan.launch_count()
    plan.forward_host(x, y, "NHWC")
    assert plan.launch_count() - before > 1
    assert rel_err(y.numpy(), ref) <= TOL["bf16"]
    plan.status()
    plan.destroy()

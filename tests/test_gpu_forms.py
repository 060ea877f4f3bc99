"""Every form of the fused bf16 forward on shapes that the default would give to another one, against the CPU reference; and the
prepared launches of one plan that serves several input sizes and options in turn."""
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
    (1, 64, 512, 9, 9, 3, 2, 1, ("heavy",)),              # few tiles, D >= 256: two blocks per tile on the ALUs
    (1, 64, 256, 9, 9, 3, 1, 1, ("uniform", 1, 3)),
    (2, 32, 512, 14, 14, 3, 1, 1, ("uniform", 1, 9)),
    (3, 16, 256, 4, 4, 3, 1, 1, ("uniform", 1, 9)),       # the same with 4-wide patches
    (2, 16, 320, 8, 8, 3, 2, 1, ("uniform", 1, 9)),
    (2, 24, 40, 20, 17, 3, 2, 1, ("uniform", 1, 9)),
    (2, 16, 24, 19, 17, 5, 2, 2, ("uniform", 1, 25)),
    (2, 40, 272, 7, 7, 1, 1, 0, ("uniform", 1, 1)),
    (20, 64, 368, 25, 24, 5, 1, 2, ("heavy",)),
    (40, 128, 128, 28, 28, 3, 1, 1, ("heavy",)),
    (16, 256, 512, 16, 16, 3, 1, 1, ("uniform", 1, 3)),   # D = 512 at several tiles per block
    (16, 128, 512, 16, 16, 3, 2, 1, ("uniform", 1, 9)),
]


@pytest.mark.parametrize("dw_math", [1, 2, 3])
@pytest.mark.parametrize("shape", SHAPES)
def test_forced_form_matches_reference(shape, dw_math):
    N, C, D, H, W, k, s, p, gd = shape
    data = gi.make_layer(small_spec("t", N, C, D, H, W, k, s, p, gd, "bf16", "NHWC", relu=(C == 24), seed=3 + sum(shape[:8])))
    ref, _ = run_oracle(data)
    assert rel_err(run_gpu(data, path=gdws.PATH_FUSED, dw_math=dw_math), ref) <= 1e-2      # two roundings to bf16


@pytest.mark.parametrize("dw_math", [1, 2, 3])
def test_one_plan_serves_sizes_and_options_in_turn(dw_math):
    sizes = [(2, 16, 16), (5, 9, 11), (1, 4, 4), (40, 16, 16)]
    layers = [gi.make_layer(small_spec("t", n, 32, 64, h, w, 3, 1, 1, ("const", 4), "bf16", "NHWC", seed=19)) for n, h, w in sizes]
    for d in layers[1:]:                                   # one set of weights
        d.dw_w, d.pw_w, d.bias = layers[0].dw_w, layers[0].pw_w, layers[0].bias
    refs = [run_oracle(d)[0] for d in layers]
    plan = make_plan(layers[0], path=gdws.PATH_FUSED, dw_math=dw_math)
    plan.pack_weights(to_device(layers[0].dw_w, "bf16"), to_device(layers[0].pw_w, "bf16"), torch.from_numpy(layers[0].bias).cuda())
    xs = [to_device(d.x, "bf16") for d in layers]
    for step in range(24):
        i, relu, f32 = step % 4, (step // 4) % 2, (step // 8) % 2
        plan.set_option(gdws.OPT_RELU, relu)
        plan.set_option(gdws.OPT_OUT_DTYPE, f32)
        yg = Guarded(refs[i].shape, torch.float32 if f32 else torch.bfloat16, fill=float("nan"))      # another buffer each time
        plan.forward(xs[i], yg.t, "NHWC")
        torch.cuda.synchronize()
        yg.check("y")
        want = np.maximum(refs[i], 0) if relu else refs[i]
        assert rel_err(yg.t.float().cpu().numpy(), want) <= 1e-2, (step, i, relu, f32)
    plan.status()
    plan.destroy()


def test_weights_given_with_a_call_of_another_form():
    """Weights that come with a call are folded only if it takes the folded form: a later call that reuses them computes with them
    and not with folded filters of earlier ones, whichever form it would have taken."""
    g = np.full(64, 2, dtype=np.int32)
    layers = [gi.make_layer(small_spec("t", n, 64, 64, h, h, 3, 1, 1, ("const", 2), "bf16", "NHWC", seed=s)) for n, h, s in ((64, 28, 5), (2, 16, 6))]
    plan = gdws.Plan(64, 64, 3, 1, 1, g)
    assert plan.form(64, 28, 28) == 3 and plan.form(2, 16, 16) == 1
    xs = [to_device(d.x, "bf16") for d in layers]
    ys = [torch.empty((d.spec.N, d.spec.Ho, d.spec.Wo, 64), dtype=torch.bfloat16, device="cuda") for d in layers]
    weights = [[to_device(d.dw_w, "bf16"), to_device(d.pw_w, "bf16"), torch.from_numpy(d.bias).cuda()] for d in layers]

    def run(i, w=None):
        ys[i].fill_(float("nan"))
        plan.forward(xs[i], ys[i], "NHWC", *(weights[w] if w is not None else []))
        torch.cuda.synchronize()
        plan.status()
        return ys[i].float().cpu().numpy()

    def want(i, w):
        d = gi.LayerData(layers[i].spec, layers[i].g, layers[i].x, layers[w].dw_w, layers[w].pw_w, layers[w].bias)
        return run_oracle(d)[0]

    plan.pack_weights(*weights[0])
    assert rel_err(run(0), want(0, 0)) <= 1e-2
    assert rel_err(run(1, 1), want(1, 1)) <= 1e-2          # two stages, other weights
    assert rel_err(run(0), want(0, 1)) <= 1e-2             # would be folded
    assert rel_err(run(0, 0), want(0, 0)) <= 1e-2          # folded, weights with the call
    assert rel_err(run(1), want(1, 0)) <= 1e-2
    plan.destroy()

"""gdws_depthwise on the tensor cores: against the ALU kernel (equal but for values next to a rounding boundary) and the CPU
oracle, bit for bit twice, padding channels zero, infinities and NaN where the ALU kernel has them.  Filters that stay and filters that
come by runs, boxes of 16, 32 and 64 channels, runs that share a box and runs of two boxes, one and several boxes per tile, both strides,
maps at most 4 wide, channels without filters."""
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


@pytest.mark.parametrize("N,C,H,W,k,stride,g", [
    (6, 64, 56, 56, 3, 1, ("uniform", 1, 4)), (3, 72, 17, 19, 3, 1, ("const", 1)), (2, 136, 15, 13, 3, 2, ("uniform", 1, 3)), (5, 40, 20, 22, 5, 1, ("uniform", 1, 25)),
    (5, 64, 7, 6, 5, 2, ("uniform", 1, 25)), (40, 72, 5, 5, 3, 2, ("uniform", 1, 3)), (9, 512, 9, 9, 3, 1, ("uniform", 1, 5)), (31, 344, 18, 15, 3, 1, ("uniform", 1, 5)),
    (4, 48, 30, 31, 3, 1, ("uniform", 0, 3)), (3, 24, 21, 20, 2, 1, ("uniform", 1, 3)), (2, 16, 9, 40, 4, 2, ("uniform", 1, 9)), (8, 88, 12, 10, 1, 1, ("uniform", 1, 2)),
])
def test_matches_alu_kernel_and_reference(N, C, H, W, k, stride, g):
    data = gi.make_layer(small_spec("t", N, C, 16, H, W, k, stride, k // 2, g, "bf16", "NHWC", seed=5 * k + C))
    s = data.spec
    plan = make_plan(data)
    plan.pack_weights(to_device(data.dw_w, "bf16"), to_device(data.pw_w, "bf16"))
    G, Gp, _, _ = plan.info()
    x = to_device(data.x, "bf16")
    zg = Guarded((N * s.Ho * s.Wo, Gp), torch.bfloat16)

    def run(dw_math):
        plan.set_option(gdws.OPT_DW_MATH, dw_math)
        assert plan.kernel(N, H, W, stage=True) == (gdws.KERNEL_GDW_TC if dw_math == 2 else gdws.KERNEL_GDW_ALU)
        zg.t.fill_(7.0)
        plan.depthwise(x, zg.t, "NHWC")
        torch.cuda.synchronize()
        plan.status()
        return zg.t.float().cpu().numpy()

    tc, alu = run(2), run(1)
    zg.check("z")
    assert np.array_equal(run(2), tc) and (tc[:, G:] == 0).all()
    _, zr, _ = run_oracle(data, return_z=True)
    assert rel_err(tc[:, :G].reshape(N, s.Ho, s.Wo, G), zr) <= 2 ** -8        # z rounded once
    differ = tc != alu                               # fp32 sums of k*k products differ in their last bits
    assert differ.mean() <= 1e-3 and np.abs(tc - alu).max() <= 2 ** -7 * np.abs(alu).max()
    flat = x.view(-1)
    for j, v in enumerate((float("inf"), float("-inf"), float("nan"))):
        flat[(j + 1) * flat.numel() // 4] = v
    tc, alu = run(2), run(1)
    for test in (np.isnan, np.isposinf, np.isneginf):
        assert np.array_equal(test(tc), test(alu))
    fine = np.isfinite(alu)
    assert not fine.all() and np.abs(tc[fine] - alu[fine]).max() <= 2 ** -7 * np.abs(alu[fine]).max()
    plan.destroy()


@pytest.mark.parametrize("v", [float("inf"), float("nan")])
@pytest.mark.parametrize("N,C,H,W,k,stride", [(64, 64, 56, 56, 3, 1), (9, 48, 41, 39, 5, 2), (20, 64, 7, 4, 3, 1)])
def test_values_that_are_not_finite_do_not_take_long(N, C, H, W, k, stride, v):
    """x that is infinite or NaN everywhere: every z is worked out again on the ALUs, as the ALU kernel has it, within some 20 times
    the time of ordinary values."""
    data = gi.make_layer(small_spec("t", N, C, 16, H, W, k, stride, k // 2, ("uniform", 1, 4), "bf16", "NHWC", seed=C + H))
    plan = make_plan(data)
    plan.pack_weights(to_device(data.dw_w, "bf16"), to_device(data.pw_w, "bf16"))
    G, Gp, _, _ = plan.info()
    x = to_device(data.x, "bf16")
    bad = torch.full_like(x, v)
    zs = [torch.full((N * data.spec.Ho * data.spec.Wo, Gp), 7.0, dtype=torch.bfloat16, device="cuda") for _ in range(2)]

    def least_ms(x):
        ms = []
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(4):
                plan.depthwise(x, zs[0], "NHWC")
            b.record()
            torch.cuda.synchronize()
            ms.append(a.elapsed_time(b))
        return min(ms)

    plan.set_option(gdws.OPT_DW_MATH, 2)
    assert plan.kernel(N, H, W, stage=True) == gdws.KERNEL_GDW_TC
    least_ms(x)
    plain, slow = least_ms(x), least_ms(bad)
    plan.set_option(gdws.OPT_DW_MATH, 1)
    plan.depthwise(bad, zs[1], "NHWC")
    torch.cuda.synchronize()
    plan.status()
    a, b = (z.float().cpu().numpy() for z in zs)
    assert np.array_equal(a, b, equal_nan=True) and not np.isfinite(a[:, :G]).all()
    assert slow <= 40 * plain
    plan.destroy()

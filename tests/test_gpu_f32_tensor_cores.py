"""The fp32 forward with its pointwise products on the tensor cores: against the CPU oracle, no less exact than the ALU kernel from 16
intermediate channels on, for values of all sizes, and with the same infinities and NaN.  Output channels around 16, 32, 64 and 128 and in two parts, chunks of 32 intermediate channels with
remainders and one alone, clusters that share a tile's chunks, tiles of several images, both filter sizes, strides, channels without filters."""
import time

import numpy as np
import pytest
import torch

from paper_2110_14871_b200 import build as gbuild
from paper_2110_14871_b200 import gdws
from paper_2110_14871_b200 import inputs as gi

from util import make_plan, rel_err, run_gpu, run_oracle, small_spec, to_device

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    gbuild.build_library()


SHAPES = [
    # N, C, D, H, W, k, stride, g
    (1, 1, 1, 5, 5, 3, 1, ("const", 1)),
    (1, 16, 16, 32, 32, 3, 1, ("uniform", 1, 3)),
    (9, 12, 33, 6, 7, 3, 1, ("uniform", 0, 9)),            # several images per tile, a channel without filters
    (16, 64, 128, 28, 28, 3, 1, ("uniform", 1, 9)),
    (2, 147, 117, 14, 10, 3, 1, ("uniform", 1, 9)),        # eight blocks per tile
    (3, 40, 200, 17, 19, 3, 2, ("uniform", 1, 9)),         # two parts of the output channels
    (5, 33, 65, 20, 22, 5, 1, ("uniform", 1, 25)),
    (2, 64, 72, 31, 22, 5, 2, ("uniform", 1, 25)),
    (400, 8, 31, 9, 9, 3, 1, ("const", 1)),                # many tiles of one chunk per block
    (2, 20, 18, 40, 300, 3, 3, ("uniform", 1, 4)),         # stride 3, long rows
]


def _on_tensor_cores(data):
    """The option falls back to the ALUs where the tensor cores do not cover a layer."""
    plan = make_plan(data, path=gdws.PATH_FUSED, dw_math=2)
    assert plan.kernel(data.spec.N, data.spec.H, data.spec.W, gdws.F32) == gdws.KERNEL_F32_PIECES
    plan.destroy()


@pytest.mark.parametrize("layout", ["NCHW", "NHWC"])
@pytest.mark.parametrize("shape", SHAPES)
def test_matches_reference(shape, layout):
    N, C, D, H, W, k, s, gd = shape
    data = gi.make_layer(small_spec("t", N, C, D, H, W, k, s, k // 2, gd, "f32", layout, relu=D == 33, seed=3 + sum(shape[:7])))
    _on_tensor_cores(data)
    ref, _ = run_oracle(data)
    tc, alu = (run_gpu(data, path=gdws.PATH_FUSED, dw_math=m) for m in (2, 1))
    # dropped products (2^-24 each) and the chunks' truncation: 2^-22 of sum |P||z|, some sqrt(G) times the largest output
    assert rel_err(tc, ref) <= 1e-5
    # one rounding per chunk instead of one per channel; both have z's own roundings.  With fewer channels than the default takes here
    # what the tensor cores truncate (2^-24 of the sum at most) can outweigh it.
    few = data.g.sum() < 16
    assert np.linalg.norm(tc - ref) <= np.linalg.norm(alu - ref) + (2 ** -24 * np.linalg.norm(ref) if few else 0.0)


@pytest.mark.parametrize("layout", ["NCHW", "NHWC"])
@pytest.mark.parametrize("N,C,D,H,W,k", [(2, 40, 40, 20, 20, 3), (1, 150, 130, 14, 10, 3), (3, 9, 20, 24, 24, 5)])
def test_nonfinite_values_are_those_of_the_sums(N, C, D, H, W, k, layout):
    data = gi.make_layer(small_spec("t", N, C, D, H, W, k, 1, k // 2, ("uniform", 1, 9), "f32", layout, seed=17 + C))
    rng = np.random.default_rng(5)
    flat = data.x.reshape(-1)
    for v in (np.inf, -np.inf, np.nan, 3.4e38):
        flat[rng.integers(0, flat.size, 3)] = v
    data.pw_w[1, 2], data.pw_w[D - 1, 0] = np.inf, 0.0
    _on_tensor_cores(data)
    got = []
    for m in (2, 1):
        got.append(run_gpu(data, path=gdws.PATH_FUSED, dw_math=m))
    for test in (np.isnan, np.isposinf, np.isneginf):
        assert np.array_equal(test(got[0]), test(got[1]))
    fine = np.isfinite(got[1])
    assert fine.any() and not fine.all()
    scale = np.abs(got[1][fine]).max()
    assert np.abs(got[0][fine] - got[1][fine]).max() <= 1e-5 * scale


@pytest.mark.parametrize("layout", ["NCHW", "NHWC"])
@pytest.mark.parametrize("N,C,D,H,W,k", [(16, 128, 128, 28, 28, 3), (1, 256, 200, 14, 15, 3), (8, 64, 40, 33, 20, 5)])
def test_an_infinite_tap_does_not_take_long(N, C, D, H, W, k, layout):
    """One tap that is infinite reaches nearly every output: those are worked out again, with the ALU kernel's infinities and NaN, in
    a time that stays near an ordinary forward's (10 to 30 times it; 1000 and more with a sum per thread)."""
    data = gi.make_layer(small_spec("t", N, C, D, H, W, k, 1, k // 2, ("uniform", 1, 9), "f32", layout, seed=9 + C))
    data.dw_w[7, 1, 1], data.dw_w[9, 0, 0] = np.inf, 3e38
    _on_tensor_cores(data)
    got = [run_gpu(data, path=gdws.PATH_FUSED, dw_math=m) for m in (2, 1)]
    for test in (np.isnan, np.isposinf, np.isneginf):
        assert np.array_equal(test(got[0]), test(got[1]))
    assert np.isfinite(got[1]).mean() < 0.1
    plan = make_plan(data, path=gdws.PATH_FUSED, dw_math=2)
    x, dw, pw = (to_device(a, "f32") for a in (data.x, data.dw_w, data.pw_w))
    y = torch.empty(got[0].shape, device="cuda")
    plain = torch.where(dw.abs() < 1e30, dw, torch.zeros_like(dw))

    def least_ms(w):
        ms = []
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            plan.forward(x, y, layout, w, pw)
            b.record()
            torch.cuda.synchronize()
            ms.append(a.elapsed_time(b))
        return min(ms)

    least_ms(plain)
    assert least_ms(dw) <= 100 * least_ms(plain)
    plan.status()
    plan.destroy()


@pytest.mark.parametrize("N,C,D,H,W,k", [(2, 40, 48, 20, 21, 3), (1, 150, 130, 14, 10, 3), (2, 17, 64, 20, 20, 5)])
def test_small_and_large_values_keep_their_bits(N, C, D, H, W, k):
    """x, taps and weights around fp32's ends: as exact as the ALU kernel, whose sums round at 2^-149 too."""
    data = gi.make_layer(small_spec("t", N, C, D, H, W, k, 1, k // 2, ("uniform", 1, 9), "f32", "NCHW", seed=31 + C))
    data.bias[:] = 0
    _on_tensor_cores(data)
    parts = [np.copy(a) for a in (data.x, data.dw_w, data.pw_w)]
    for ends in [(0, 0, -60), (-60, 0, 0), (-60, -30, -20), (0, 0, -100), (0, 0, -110), (0, 0, -116), (0, 0, -123), (-100, 0, 0), (-110, 0, 0), (-116, 0, 0), (-123, 0, 0), (0, -123, 0), (-123, 100, 0), (60, 0, -123),
                 (0, 0, 40), (40, 20, 30), (100, 0, 0), (0, 110, 0), (0, 0, 110), (0, 60, 50)]:
        for a, p, e in zip((data.x, data.dw_w, data.pw_w), parts, ends):
            a[...] = np.ldexp(p, e)
        ref, _ = run_oracle(data)
        tc, alu = (run_gpu(data, path=gdws.PATH_FUSED, dw_math=m) for m in (2, 1))
        size = np.linalg.norm(np.ldexp(ref, -sum(ends)))         # in range for its squares
        err = [np.linalg.norm(np.ldexp(y - ref, -sum(ends))) / size for y in (tc, alu)]
        assert err[0] <= err[1] and err[0] <= 1e-5, (ends, err)


def test_a_repeated_call_does_no_work_per_filter_on_the_host():
    """G = 262144: what a launch needs is worked out with the first call of a size (a pass over the filters takes 250 us)."""
    data = gi.make_layer(small_spec("t", 1, 64, 8, 6, 6, 3, 1, 1, ("const", 4096), "f32", "NCHW", seed=5))
    plan = make_plan(data, path=gdws.PATH_FUSED, dw_math=2)
    assert plan.kernel(1, 6, 6, gdws.F32) == gdws.KERNEL_F32_PIECES
    x, dw, pw = (to_device(a, "f32") for a in (data.x, data.dw_w, data.pw_w))
    y = torch.empty((1, 8, 6, 6), device="cuda")
    us = []
    for _ in range(8):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        plan.forward(x, y, "NCHW", dw, pw)
        us.append(1e6 * (time.perf_counter() - t0))
    plan.status()
    plan.destroy()
    assert min(us) <= 80, us

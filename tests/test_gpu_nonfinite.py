"""Infinities and NaN in x: they reach the outputs that the operator's sums connect them with, with the value of those sums,
and no others."""
import numpy as np
import pytest

from paper_2110_14871_b200 import build as gbuild
from paper_2110_14871_b200 import gdws
from paper_2110_14871_b200 import inputs as gi

from util import run_gpu, small_spec

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    gbuild.build_library()


# channel counts whose G is no multiple of the kernels' chunks; tiles below and above 32 pixels, filter sizes with and without code of their own
@pytest.mark.parametrize("layout", ["NCHW", "NHWC"])
@pytest.mark.parametrize("N,C,D,H,W,k", [(1, 3, 16, 8, 8, 3), (2, 5, 40, 40, 40, 3), (6, 9, 128, 56, 56, 3), (2, 5, 20, 24, 24, 5), (1, 3, 16, 9, 9, 2), (8, 7, 128, 40, 40, 1)])
def test_f32_infinity_in_the_last_channel(N, C, D, H, W, k, layout):
    data = gi.make_layer(small_spec("t", N, C, D, H, W, k, 1, k // 2, ("const", 1), "f32", layout, seed=41 + C))
    data.x[...] = np.abs(data.x)
    data.dw_w[...] = np.abs(data.dw_w) + 0.1        # every window that holds the infinity sums to +infinity
    data.pw_w[...] = np.abs(data.pw_w) + 0.1
    at = (0, C - 1, H // 2, W // 2) if layout == "NCHW" else (0, H // 2, W // 2, C - 1)
    data.x[at] = np.inf
    y = run_gpu(data, path=gdws.PATH_FUSED)
    y = y if layout == "NCHW" else np.moveaxis(y, 3, 1)
    s = data.spec
    want = np.zeros((N, s.Ho, s.Wo), dtype=bool)
    lo = s.pad - k + 1                                # output rows h with h - pad <= H // 2 < h - pad + k
    want[0, max(0, H // 2 + lo):H // 2 + s.pad + 1, max(0, W // 2 + lo):W // 2 + s.pad + 1] = True
    assert not np.isnan(y).any()
    assert np.array_equal(np.isposinf(y), np.broadcast_to(want[:, None], y.shape))


@pytest.mark.parametrize("C,D,H,k,stride", [(24, 40, 20, 3, 1), (136, 72, 9, 3, 2), (64, 64, 16, 5, 1)])
def test_bf16_unused_channel_is_not_read(C, D, H, k, stride):
    """A channel with g_c = 0 is no part of the layer, whatever it holds: layers whose GDW stage runs on the ALUs by default."""
    data = gi.make_layer(small_spec("t", 3, C, D, H, H + 1, k, stride, k // 2, ("const", 2), "bf16", "NHWC", seed=43))
    data.g[5] = 0
    G = int(data.g.sum())
    data.dw_w, data.pw_w = data.dw_w[:G], np.ascontiguousarray(data.pw_w[:, :G])
    want = run_gpu(data, path=gdws.PATH_FUSED)
    for v in (np.inf, np.nan):
        data.x[..., 5] = v
        assert np.array_equal(run_gpu(data, path=gdws.PATH_FUSED), want) and np.isfinite(want).all()

"""The folded form of layers with up to 48 input channels on pairs of SMs: one window of one to three K steps, both filter sizes,
filters with and without their second term."""
import numpy as np
import pytest
import torch

from paper_2110_14871_b200 import build as gbuild
from paper_2110_14871_b200 import gdws
from paper_2110_14871_b200 import inputs as gi

from util import rel_err, run_gpu, run_oracle, small_spec

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    gbuild.build_library()


@pytest.mark.parametrize("zero_sum", [False, True])
@pytest.mark.parametrize("C,D,k", [(8, 40, 3), (16, 16, 5), (24, 72, 3), (32, 136, 5), (40, 24, 3), (48, 64, 3), (48, 32, 5), (56, 48, 3)])
def test_narrow_layers_match_reference(C, D, k, zero_sum):
    data = gi.make_layer(small_spec("t", 3, C, D, 86, 97, k, 1, k // 2, ("uniform", 1, 3), "bf16", "NHWC", relu=C == 24, seed=C + D))      # 3 x 6 x 13 tiles
    if zero_sum:
        data.dw_w[...] = torch.from_numpy(data.dw_w - data.dw_w.mean(axis=(1, 2), keepdims=True)).to(torch.bfloat16).float().numpy()
    y = run_gpu(data, path=gdws.PATH_FUSED, dw_math=3, prepack=True)
    assert rel_err(y, run_oracle(data)[0]) <= 1e-2         # folded filters and y rounded once each: 2^-8 and 2^-9, and sums
    assert np.array_equal(run_gpu(data, path=gdws.PATH_FUSED, dw_math=3, prepack=True), y)

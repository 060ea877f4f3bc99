"""The fp32 forward at the edges of its block tiles: pixel runs that end inside a tile and cross image rows and images,
output channels around 16, 32, 64 and 128, K chunks of 16 with remainders, channels without filters, strides and filter sizes.
Reference: the CPU oracle in fp64; fp32 sums of up to 10^4 terms stay within 1e-5 of the largest output (2^-24 * sqrt(terms))."""
import pytest

from paper_2110_14871_b200 import build as gbuild
from paper_2110_14871_b200 import gdws
from paper_2110_14871_b200 import inputs as gi

from util import rel_err, run_gpu, run_oracle, small_spec

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    gbuild.build_library()


SHAPES = [
    # N, C, D, H, W, k, stride, pad, g_dist
    (1, 1, 1, 1, 1, 3, 1, 1, ("const", 1)),
    (7, 3, 17, 5, 3, 3, 1, 1, ("uniform", 0, 9)),          # rows of 3: a tile crosses many rows and images
    (2, 40, 33, 31, 29, 3, 2, 1, ("uniform", 0, 2)),
    (1, 33, 129, 40, 41, 3, 1, 1, ("uniform", 1, 9)),
    (6, 16, 128, 56, 56, 3, 1, 1, ("uniform", 1, 3)),      # the widest tiles
    (40, 24, 100, 28, 28, 3, 1, 1, ("const", 2)),
    (2, 6, 40, 30, 23, 5, 1, 2, ("uniform", 1, 25)),
    (3, 5, 20, 17, 19, 7, 2, 3, ("uniform", 1, 20)),       # any-size filter code
    (2, 9, 24, 21, 18, 2, 3, 0, ("uniform", 1, 4)),        # stride beyond the filter
    (2, 8, 16, 20, 20, 4, 4, 2, ("const", 3)),
    (3, 70, 64, 9, 9, 1, 1, 0, ("uniform", 1, 1)),
]


@pytest.mark.parametrize("layout", ["NCHW", "NHWC"])
@pytest.mark.parametrize("shape", SHAPES)
def test_f32_tiles_match_reference(shape, layout):
    N, C, D, H, W, k, s, p, gd = shape
    spec = small_spec("t", N, C, D, H, W, k, s, p, gd, "f32", layout, relu=(C % 2 == 0), seed=5 + sum(shape[:8]))
    data = gi.make_layer(spec)
    ref, _ = run_oracle(data)
    assert rel_err(run_gpu(data, path=gdws.PATH_FUSED), ref) <= 1e-5

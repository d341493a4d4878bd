"""Second pass of the fused layer at the edges of its tiling: both CTA shapes, K ranges that are built in parts, several
chunks of output channels, ragged tiles and channel counts.  Comparison and tolerances are those of the layer tests."""
import pytest

from paper_2205_12268_b200 import inputs
from test_gpu_layer import _run_and_compare, wcc      # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

SHAPES = [  # N, Cin, Cout, H, W, dtype, levels, gamma, bits
    (3, 21, 37, 224, 244, "f32", 2, 0.2, 8),          # more tile groups than SMs: two CTAs per SM; two chunks, ragged width
    (3, 10, 34, 240, 248, "bf16", 3, 0.3, 0),         # the same without quantization
    (11, 130, 30, 96, 152, "bf16", 3, 0.2, 8),        # two CTAs per SM, K in two parts, one chunk
    (1, 225, 67, 32, 72, "bf16", 3, 0.4, 8),          # one CTA per SM, K in two parts, rebuilt for a second chunk
    (1, 9, 1000, 16, 40, "f32", 3, 0.5, 8),           # many chunks, the last one ragged
    (2, 230, 16, 128, 256, "bf16", 2, 0.1, 0),        # fifteen K steps of bf16 in three parts
    (2, 19, 35, 18, 22, "bf16", 1, 0.5, 8),           # rows of 4m + 2 elements
    (2, 7, 65, 10, 30, "f32", 1, 0.5, 0),
]


@pytest.mark.parametrize("cfg", SHAPES, ids=lambda c: "N%d_%dto%d_%dx%d_%s_L%d_g%s_b%d" % c)
def test_second_pass(wcc, cfg):                       # noqa: F811
    N, Cin, Cout, H, W, dtype, L, gamma, bits = cfg
    _run_and_compare(wcc, inputs.custom("pass2", 4, N, Cin, Cout, H, W, dtype, L, gamma, bits, n_sin=4, fmax=3.0))

"""The pipeline around the gathered columns on rows of 4m + 2 elements (one level), with a convolution in front and without:
last lane with one quad, fewer columns than a tile, channel counts around the chunks of sixteen and eight."""
import pytest

import test_gpu_block as block
from test_gpu_layer import wcc      # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

LAYERS = [  # N, Cin, Cout, H, W, dtype, levels, gamma, bits
    (2, 300, 70, 12, 30, "f32", 1, 0.5, 8),
    (1, 271, 193, 10, 130, "bf16", 1, 0.4, 8),
    (3, 224, 79, 24, 22, "bf16", 1, 0.0625, 6),
    (1, 200, 105, 18, 46, "bf16", 1, 0.3, 0),
    (2, 265, 66, 4, 6, "f32", 1, 0.6, 0),
]


@pytest.mark.parametrize("cfg", LAYERS, ids=lambda c: "N%d_%dto%d_%dx%d_%s_L%d_g%s_b%d" % c)
def test_layer(wcc, cfg):      # noqa: F811
    block.test_wide_layer_without_coefficient_map(wcc, cfg)


@pytest.mark.parametrize("cfg", [(2, 20, 72, 12, 30, "f32", 1, 0.5), (1, 9, 33, 10, 134, "bf16", 1, 0.25), (1, 17, 40, 4, 2, "bf16", 1, 0.5)],
                         ids=lambda c: "N%d_c%d_e%d_%dx%d_%s_L%d_g%s" % c)
def test_block(wcc, cfg):      # noqa: F811
    block.test_inverted_residual_block(wcc, cfg)

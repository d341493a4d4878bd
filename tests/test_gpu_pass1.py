"""Forward transform and norms with one, two, four and eight warps per tile (chosen from the tile count), channel counts
around a box and rounds that leave warps idle: coefficients and norms equal the oracle's bit for bit."""
import numpy as np
import pytest
import torch

import oracle
from paper_2205_12268_b200 import inputs
from test_gpu_layer import wcc      # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

SHAPES = [  # N, C, H, W, levels  (tiles of 256 positions)
    (1, 1, 8, 8, 3), (1, 3, 4, 6, 1), (1, 9, 16, 40, 3), (2, 70, 24, 72, 2),          # eight warps
    (3, 17, 128, 256, 3), (5, 8, 96, 150, 1),                                         # four
    (6, 33, 128, 256, 2),                                                             # two
    (10, 5, 128, 264, 3),                                                             # one
    (14, 9, 128, 256, 2),                                                             # two again: more than one wave
    (19, 12, 128, 256, 3),                                                            # two (bf16), four (fp32)
    (24, 9, 128, 256, 1),                                                             # one again: several waves
]


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("shape", SHAPES, ids=str)
def test_transform_and_norms(wcc, shape, dtype):      # noqa: F811
    N, C, H, W, L = shape
    x = inputs.feature_map(11, N, C, H, W, 4, 3.0).astype(np.float32)
    if dtype == "bf16":
        b = inputs.f32_to_bf16_bits(x)
        x, xd = inputs.bf16_bits_to_f32(b), torch.from_numpy(b.view(np.int16)).cuda().view(torch.bfloat16)
    else:
        xd = torch.from_numpy(x).cuda()
    coef, nrm2 = wcc.haar_fwd(xd, L)
    assert wcc.last_status() == 0
    want_c = oracle.haar_fwd(x, L)
    want_n = oracle.norms(want_c)
    assert np.array_equal(coef.cpu().numpy().view(np.uint32).reshape(-1), want_c.view(np.uint32).reshape(-1))
    assert np.array_equal(nrm2.cpu().numpy().view(np.uint32).reshape(-1), want_n.view(np.uint32).reshape(-1))

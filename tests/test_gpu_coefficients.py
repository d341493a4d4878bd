"""Coefficients stored with the channels split over the grid (many channels, or rows of 4m + 2), with and without a convolution in
front: chunks of four that leave a remainder, the last channel, ragged tiles.  Bit for bit the oracle's."""
import numpy as np
import pytest
import torch

import oracle
from paper_2205_12268_b200 import inputs
from test_gpu_layer import wcc      # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

SHAPES = [  # N, C, H, W, levels
    (1, 97, 4, 6, 1), (2, 131, 12, 30, 1), (1, 259, 6, 10, 1), (1, 514, 2, 2, 1),         # rows of 4m + 2
    (3, 35, 400, 10, 1),                                                                   # the same, few channels on 600 tiles
    (1, 101, 8, 8, 3), (2, 263, 8, 72, 2), (1, 1030, 16, 40, 3),
    (4, 259, 300, 8, 1), (4, 98, 600, 4, 1), (20, 261, 64, 32, 3),                         # from one, four and eight tiles per SM on
    (4, 7, 600, 8, 1), (4, 30, 600, 10, 1), (2, 16, 40, 22, 1), (10, 9, 512, 32, 2),       # all channels by one warp
]


def _bits(a):
    return np.ascontiguousarray(a, dtype=np.float32).view(np.uint32).reshape(-1)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("shape", SHAPES, ids=str)
def test_transforms(wcc, shape, dtype):      # noqa: F811
    N, C, H, W, L = shape
    x = inputs.feature_map(7, N, C, H, W, 2, 3.0).astype(np.float32)
    k9 = np.random.default_rng(4).standard_normal((C, 3, 3)).astype(np.float32)
    if dtype == "bf16":
        b = inputs.f32_to_bf16_bits(x)
        x, xd = inputs.bf16_bits_to_f32(b), torch.from_numpy(b.view(np.int16)).cuda().view(torch.bfloat16)
    else:
        xd = torch.from_numpy(x).cuda()
    for got, want in ((wcc.haar_fwd(xd, L), oracle.haar_fwd(x, L)),
                      (wcc.dwconv_haar_fwd(xd, torch.from_numpy(k9).cuda(), L), oracle.haar_fwd(oracle.dwconv3x3(x, k9), L))):
        assert np.array_equal(_bits(got[0].cpu().numpy()), _bits(want))
        assert np.array_equal(_bits(got[1].cpu().numpy()), _bits(oracle.norms(want)))
    back = wcc.haar_inv(torch.from_numpy(oracle.haar_fwd(x, L)).cuda(), L)
    assert torch.equal(back.cpu(), torch.from_numpy(oracle.haar_inv(oracle.haar_fwd(x, L), L)))
    assert wcc.last_status() == 0

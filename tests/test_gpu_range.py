"""The public transforms over the whole range of their types: coefficients and norms are those of Eq. 3 with its halvings, for
maps whose sums would overflow without them, whose squares are near the ends of fp32 and which are subnormal."""
import numpy as np
import pytest
import torch

import oracle
from paper_2205_12268_b200 import inputs
from test_gpu_layer import wcc      # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def _bits(a):
    return np.ascontiguousarray(a, dtype=np.float32).view(np.uint32).reshape(-1)


@pytest.mark.parametrize("exponent", [59, 123, -64, -72, -130])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("shape", [(1, 3, 16, 40, 3), (2, 9, 8, 36, 2), (1, 5, 6, 30, 1)], ids=str)
def test_transforms(wcc, shape, dtype, exponent):      # noqa: F811
    N, C, H, W, L = shape
    x = (inputs.feature_map(5, N, C, H, W, 4, 3.0).astype(np.float32) * np.float32(2.0) ** np.float32(exponent)).astype(np.float32)
    k9 = np.random.default_rng(3).standard_normal((C, 3, 3)).astype(np.float32) / np.float32(8)
    if dtype == "bf16":
        b = inputs.f32_to_bf16_bits(x)
        x, xd = inputs.bf16_bits_to_f32(b), torch.from_numpy(b.view(np.int16)).cuda().view(torch.bfloat16)
    else:
        xd = torch.from_numpy(x).cuda()
    for got, want in ((wcc.haar_fwd(xd, L), oracle.haar_fwd(x, L)),
                      (wcc.dwconv_haar_fwd(xd, torch.from_numpy(k9).cuda(), L), oracle.haar_fwd(oracle.dwconv3x3(x, k9), L))):
        assert np.array_equal(_bits(got[0].cpu().numpy()), _bits(want))
        assert np.array_equal(_bits(got[1].cpu().numpy()), _bits(oracle.norms(want)))
    assert wcc.last_status() == 0

"""Both forms of a block's second layer: coefficients stored (at least 600 expanded channels in fp32, or on many tiles) and gathered
from a second transform, chosen by shape and by the scratch at hand."""
import pytest
import torch

import test_gpu_block as block
from test_gpu_layer import wcc      # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cfg", [(1, 20, 600, 8, 24, "f32", 3, 0.25), (2, 12, 601, 12, 20, "f32", 2, 0.5), (20, 6, 606, 32, 8, "bf16", 1, 0.25),
                                 (1, 16, 599, 16, 24, "f32", 3, 0.25)], ids=lambda c: "N%d_c%d_e%d_%dx%d_%s_L%d_g%s" % c)
def test_block(wcc, cfg):      # noqa: F811
    block.test_inverted_residual_block(wcc, cfg)


def test_less_scratch_same_result(wcc):      # noqa: F811
    """The scratch of a smaller block of the same layer does for the form that stores nothing."""
    N, C, E, H, W = 4, 32, 640, 64, 64
    g = torch.Generator(device="cuda").manual_seed(5)
    x = torch.randn((N, C, H, W), device="cuda", generator=g)
    w = [torch.randn(s, device="cuda", generator=g) / 8 for s in ((E, C), (E, 3, 3), (C, E))]
    b = wcc.Block(x, *w, 3, H * W // 4, 8)
    want = b(x)
    less = wcc.Workspace(b.ws.nbytes - N * E * H * W * 2, x.device)            # half of the coefficient map is missing
    b.ws = less
    assert torch.equal(b(x), want)
    assert wcc.last_status() == 0

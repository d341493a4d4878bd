"""Weights quantized ahead of the call on layers of many channels: K in several parts, many chunks of output channels; the same bytes
as the layer that quantizes them itself."""
import pytest
import torch

from test_gpu_layer import wcc      # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cfg", [(2, 300, 70, 16, 32, 3), (1, 1030, 520, 16, 24, 2), (1, 64, 6000, 8, 16, 3), (2, 8192, 33, 4, 10, 1), (1, 700, 40, 64, 128, 3)],
                         ids=lambda c: "N%d_%dto%d_%dx%d_L%d" % c)
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16], ids=["f32", "bf16"])
def test_same_as_quantized_by_the_layer(wcc, cfg, dtype):      # noqa: F811
    N, Cin, Cout, H, W, L = cfg
    g = torch.Generator(device="cuda").manual_seed(Cin)
    x = torch.randn((N, Cin, H, W), device="cuda", generator=g).to(dtype)
    Wt = torch.randn((Cout, Cin), device="cuda", generator=g)
    want, t = wcc.forward(x, Wt, L, H * W // 4, 8, taps=("Wq", "scale_w"))
    assert torch.equal(wcc.forward(x, None, L, H * W // 4, 8, Wq=t["Wq"], scale_w=t["scale_w"]), want)
    assert wcc.last_status() == 0

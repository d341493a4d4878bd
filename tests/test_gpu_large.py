"""Maps and matrices beyond 32-bit offsets.  Each case allocates most of a B200's memory and is skipped where it is not free."""
import pytest
import torch

from test_gpu_layer import wcc      # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def _need(gib):
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < gib << 30:
        pytest.skip("needs %d GiB of free device memory" % gib)


def test_accumulators_beyond_64_gib(wcc):      # noqa: F811
    """17 images of 131072 positions, all kept, 8192 output channels: 68 GiB of accumulators in rows of 32 KiB.  Integers in:
    without quantization the layer is the dense product, exactly (at most 16 * 24 * 2 = 96 * 8 in magnitude)."""
    _need(120)
    N, Cin, Cout, H, W = 17, 16, 8192, 256, 512
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randint(-3, 4, (N, Cin, H, W), device="cuda", generator=g).to(torch.bfloat16) * 8
    Wt = torch.randint(-2, 3, (Cout, Cin), device="cuda", generator=g).float()
    y = wcc.forward(x, Wt, 1, H * W, 0)
    assert wcc.last_status() == 0
    for n in (0, 8, N - 1):
        flat = x[n].float().reshape(Cin, -1)
        for o in range(0, Cout, 1024):
            assert torch.equal(y[n, o:o + 1024].reshape(1024, -1).float(), Wt[o:o + 1024] @ flat), (n, o)
    del x, y
    torch.cuda.empty_cache()

"""Second pass of the fused layer at the edges of its tiling: both CTA shapes, K ranges that are built in parts, several
chunks of output channels, ragged tiles and channel counts.  Comparison and tolerances are those of the layer tests."""
import pytest
import torch

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


# One launch or two, and how the last groups are shared.  Plain calls against calls with taps, which take one launch of sixteen warps
# per group and are compared with the oracle by the tests above: the same integers, so the same bits.
SPLITS = [
    (3, 12, 20, 400, 256, "f32", 2, 0.2),             # 300 groups: 296 by one launch, 4 by the next
    (9, 40, 24, 132, 376, "bf16", 2, 0.3),            # 446: 150 more than two for every SM, so one launch
    (5, 10, 50, 440, 272, "bf16", 3, 0.1),            # 619: two waves and 27 groups
    (4, 9, 12, 216, 360, "f32", 3, 0.25),             # 324 with a ragged width
    # the same with channels enough for two launches (the four above are too light for it)
    (3, 12, 100, 400, 256, "f32", 2, 0.2),
    (9, 140, 24, 132, 376, "bf16", 2, 0.3),
    (5, 110, 50, 440, 272, "bf16", 3, 0.1),
    (4, 57, 12, 216, 360, "f32", 3, 0.25),
    (1, 20, 70, 60, 92, "bf16", 2, 0.25),             # 80 padded channels on few groups: shares of 16
    (2, 33, 112, 64, 128, "f32", 3, 0.25),            # seven units of sixteen
    (3, 24, 200, 96, 160, "bf16", 3, 0.25),           # thirteen units among three CTAs: the last one has fewer
]


@pytest.mark.parametrize("cfg", SPLITS, ids=lambda c: "N%d_%dto%d_%dx%d_%s_L%d_g%s" % c)
def test_launches_and_shares(wcc, cfg):               # noqa: F811
    N, Cin, Cout, H, W, dtype, L, gamma = cfg
    gen = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn((N, Cin, H, W), device="cuda", generator=gen).to(torch.bfloat16 if dtype == "bf16" else torch.float32)
    Wt = torch.randn((Cout, Cin), device="cuda", generator=gen)
    W2 = torch.randn((Cin, Cout), device="cuda", generator=gen)
    k = inputs.keep_count(gamma, H * W)
    want, _ = wcc.forward(x, Wt, L, k, 8, taps=("Xq", "acc"))
    for _ in range(2):
        assert torch.equal(wcc.forward(x, Wt, L, k, 8, y=torch.full_like(want, 7.0)), want)
    # a layer behind it starts only when both launches are complete
    relu = torch.relu(want)
    want2, _ = wcc.forward(relu, W2, L, k, 8, taps=("Xq", "acc"))
    assert torch.equal(wcc.Chain(x, [Wt, W2], L, k, 8)(x), want2)
    assert wcc.last_status() == 0


def _map_of_groups(groups):
    """N, H, W of a batch that the second pass runs as this many groups at two levels (tiles of 4 x 64, four to a group)."""
    for N in range(5, 25):
        for w in range(8, 1, -1):
            for h in range(90, 8, -1):
                if -(-N * w * h // 4) == groups and 4 * h * 64 * w <= 131072:
                    return N, 4 * h, 64 * w
    raise AssertionError(groups)


@pytest.mark.parametrize("opts", ["plain", "residual", "alpha", "bits0"])
@pytest.mark.parametrize("last", [lambda sms: 1, lambda sms: 100, lambda sms: sms - 1, lambda sms: sms, lambda sms: sms + 1],
                         ids=["1", "100", "sms-1", "sms", "sms+1"])
def test_last_groups(wcc, last, opts):                # noqa: F811
    """Heavy groups (fp32, 16 -> 96 channels): last waves up to the size that is a launch of its own (one group per SM) and one beyond,
    shared among SMs and not, with every kind of option; the call with taps is one launch.  Sixteen input channels: one K step, so
    unquantized sums have one order too."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    N, H, W = _map_of_groups(2 * sms + last(sms))
    gen = torch.Generator(device="cuda").manual_seed(5)
    x = torch.randn((N, 16, H, W), device="cuda", generator=gen)
    Wt = torch.randn((96, 16), device="cuda", generator=gen)
    kw = dict(plain={}, residual=dict(residual=torch.randn((N, 96, H, W), device="cuda", generator=gen), relu=True),
              alpha=dict(alpha=2.0), bits0={})[opts]
    k, bits = inputs.keep_count(0.25, H * W), 0 if opts == "bits0" else 8
    want, _ = wcc.forward(x, Wt, 2, k, bits, taps=("Xb" if bits == 0 else "Xq", "acc"), **kw)
    ws = wcc.Workspace.for_problem(x, 96, 2, k, bits)
    for i in range(3):                                 # the workspace of the calls before holds their words
        assert torch.equal(wcc.forward(x, Wt, 2, k, bits, y=torch.full_like(want, 7.0), ws=ws, **kw), want)
    assert wcc.last_status() == 0

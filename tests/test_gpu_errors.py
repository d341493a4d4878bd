"""A launch that the runtime rejects is an error of the call that made it and of no later one."""
import pytest
import torch

from test_gpu_layer import wcc      # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def test_rejected_launch_leaves_no_error_behind(wcc):      # noqa: F811
    x = torch.zeros((65536, 1, 2, 2), device="cuda")                   # one image more than a grid has rows
    one = torch.ones((1, 1), device="cuda")
    with pytest.raises(wcc.WccError) as e:
        wcc.forward(x, one, 1, 1, 8, staged=True)
    assert e.value.code == 8
    small = torch.ones((1, 1, 8, 8), device="cuda")
    assert torch.equal(wcc.forward(small, one, 1, 64, 0), small)
    assert wcc.last_status() == 0

"""The strided pixel copy ahead of a strided 1x1 layer: rows of one unit, of exactly one block's share, of several, every stride and type."""
import pytest
import torch

import paper_2012_00596_b200 as npas

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("stride", [1, 2, 3])
@pytest.mark.parametrize("N,H,W,C", [(1, 1, 1, 8), (3, 9, 7, 24), (2, 5, 32, 256), (1, 3, 33, 512), (2, 2, 65, 1032), (70, 4, 4, 64)])
def test_subsample_copies_every_row(N, H, W, C, stride, dtype):
    x = torch.randn((N, H, W, C), generator=torch.Generator().manual_seed(7)).to(dtype).cuda()
    x.mul_(2)                                                   # (a kernel of the same stream right ahead of the call)
    assert torch.equal(npas.subsample2d(x, stride), x[:, ::stride, ::stride, :].contiguous())

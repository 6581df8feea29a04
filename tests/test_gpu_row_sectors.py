"""Epilogues that write 32 bytes of a row at once: outputs and residuals on and off 32-byte boundaries give the same bytes."""
import pytest
import torch

import paper_2012_00596_b200 as npas
from paper_2012_00596_b200 import inputs
from util import dev

pytestmark = pytest.mark.gpu


def _at(t, byte_offset):
    """A copy of t that starts `byte_offset` bytes behind a 256-byte boundary."""
    buf = torch.empty(t.numel() * t.element_size() + 512, dtype=torch.uint8, device="cuda")
    start = (-buf.data_ptr()) % 256 + byte_offset
    v = buf[start:start + t.numel() * t.element_size()].view(t.dtype).view(t.shape)
    return v.copy_(t)


@pytest.mark.parametrize("out_dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("path,variant", [(6, 0), (7, 0), (7, 1 << 24), (8, 0)])
def test_conv_outputs_off_a_sector(path, variant, out_dtype):
    c = inputs.conv_case(dtype="bf16", residual=True, seed=313, N=3, H=14, W=13, C=64, K=64, Mb=16, Nb=16, keep=3)
    x, blob, bias = dev(c.x, "bf16"), npas.pack_bp(dev(c.w, "bf16"), c.tap_mask, 16, 16), dev(c.bias)
    res = dev(c.residual).to(out_dtype)
    kw = dict(relu=c.relu, out_dtype=out_dtype, path=path, variant=variant)
    want = npas.conv2d_bp(x, blob, bias, res, **kw)
    for y_off, r_off in ((16, 0), (0, 16), (16, 16), (48, 32)):
        y = _at(torch.zeros_like(want), y_off)
        npas.conv2d_bp(x, blob, bias, _at(res, r_off), out=y, **kw)
        assert torch.equal(y, want), (y_off, r_off)


@pytest.mark.parametrize("path", [5, 6])
def test_gemm_outputs_off_a_sector(path):
    c = inputs.config3(M=300)
    x, blob, bias = dev(c.x, "bf16"), npas.pack_bb(dev(c.w, "bf16"), c.row_keep, c.col_keep, 64, 64), dev(c.bias)
    res = torch.randn((300, c.w.shape[0]), device="cuda")
    kw = dict(relu=True, out_dtype=torch.float32, path=path)
    want = npas.linear_bb(x, blob, bias, res, **kw)
    for y_off, r_off in ((16, 0), (0, 16), (16, 16)):
        y = _at(torch.zeros_like(want), y_off)
        npas.linear_bb(x, blob, bias, _at(res, r_off), out=y, **kw)
        assert torch.equal(y, want), (y_off, r_off)

"""Column tiles that do not divide the output width: the last tile narrower, on CTAs and on CTA pairs, staged and direct stores."""
import pytest
import torch

import oracle
import paper_2012_00596_b200 as npas
from paper_2012_00596_b200 import inputs
from util import TOL_BF16, dev, floored_rel_err, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("path,bn", [(5, 64), (5, 128), (5, 192), (5, 256), (6, 128), (6, 192), (6, 256), (0, 0)])
@pytest.mark.parametrize("M,I,O", [(131, 64, 320), (1000, 192, 640), (5000, 128, 896), (257, 320, 384)])
def test_ragged_column_tiles(M, I, O, path, bn):
    if path == 6 and O % 128:
        pytest.skip("pairs take widths that 128 divides")
    c = inputs.linear_case(M=M, I=I, O=O, Bo=64, Bi=64, keep_rows=32, keep_cols=48, dtype="bf16", seed=1401)
    r = torch.randn(M, O, generator=torch.Generator().manual_seed(9)).to(torch.bfloat16)
    blob, ws = npas.pack_bb(dev(c.w, "bf16"), c.row_keep, c.col_keep, c.Bo, c.Bi), npas.workspace()
    ref = oracle.linear_bb(c.x, c.w, c.row_keep, c.col_keep, Bo=c.Bo, Bi=c.Bi, bias=c.bias, residual=r.double().numpy(), relu=c.relu)
    for odt in (torch.bfloat16, torch.float32):
        f = lambda: npas.linear_bb(dev(c.x, "bf16"), blob, dev(c.bias), r.to(odt).cuda(), relu=c.relu,
                                   out_dtype=odt, ws=ws, path=path, variant=bn)
        y = f()
        npas.check_device_status(ws)
        assert floored_rel_err(host(y), ref) < TOL_BF16
        assert torch.equal(y, f())


@pytest.mark.parametrize("bn", [16, 32, 48, 80, 112, 128, 144, 192, 240, 256])
@pytest.mark.parametrize("M,O", [(300, 1000), (129, 24)])
def test_requested_tiles_where_16_does_not_divide_the_outputs(M, O, bn):
    c = inputs.linear_case(M=M, I=192, O=O, Bo=8, Bi=64, keep_rows=5, keep_cols=48, dtype="bf16", seed=1402)
    r = torch.randn(M, O, generator=torch.Generator().manual_seed(9)).to(torch.bfloat16)
    blob, ws = npas.pack_bb(dev(c.w, "bf16"), c.row_keep, c.col_keep, c.Bo, c.Bi), npas.workspace()
    ref = oracle.linear_bb(c.x, c.w, c.row_keep, c.col_keep, Bo=c.Bo, Bi=c.Bi, bias=c.bias, residual=r.double().numpy(), relu=c.relu)
    for odt in (torch.bfloat16, torch.float32):
        y = torch.full((M, O), float("nan"), dtype=odt, device="cuda")          # every element is written
        npas.linear_bb(dev(c.x, "bf16"), blob, dev(c.bias), r.to(odt).cuda(), relu=c.relu, out=y, ws=ws, path=5, variant=bn)
        npas.check_device_status(ws)
        assert floored_rel_err(host(y), ref) < TOL_BF16


@pytest.mark.parametrize("M,I,O", [(5000, 512, 1008), (20000, 64, 80), (3000, 256, 2000), (9000, 128, 48), (300, 1024, 16), (12000, 192, 208)])
def test_widths_that_only_16_divides(M, I, O):
    """Automatic column tiles there: a multiple of 64 with the last one cut, or a power of two."""
    c = inputs.linear_case(M=M, I=I, O=O, Bo=16, Bi=64, keep_rows=8, keep_cols=48, dtype="bf16", seed=1403)
    r = torch.randn(M, O, generator=torch.Generator().manual_seed(9)).to(torch.bfloat16)
    blob, ws = npas.pack_bb(dev(c.w, "bf16"), c.row_keep, c.col_keep, c.Bo, c.Bi), npas.workspace()
    ref = oracle.linear_bb(c.x, c.w, c.row_keep, c.col_keep, Bo=c.Bo, Bi=c.Bi, bias=c.bias, residual=r.double().numpy(), relu=c.relu)
    for odt in (torch.bfloat16, torch.float32):
        for path in (0, 5):
            y = torch.full((M, O), float("nan"), dtype=odt, device="cuda")
            npas.linear_bb(dev(c.x, "bf16"), blob, dev(c.bias), r.to(odt).cuda(), relu=c.relu, out=y, ws=ws, path=path)
            npas.check_device_status(ws)
            assert floored_rel_err(host(y), ref) < TOL_BF16

"""Split-input form of the dense-image GEMM (few output tiles, a cluster of CTAs per tile) and ragged widths: column
counts that 16 does not divide, input widths that 64 does not divide, single rows, tile edges."""
import pytest
import torch

import oracle
import paper_2012_00596_b200 as npas
from paper_2012_00596_b200 import inputs
from util import TOL_BF16, TOL_F32, dev, floored_rel_err, host

pytestmark = pytest.mark.gpu


def _run(M, I, O, Bo, Bi, variant=0, path=0, out_dtype=None, res=False, seed=901):
    c = inputs.linear_case(M=M, I=I, O=O, Bo=Bo, Bi=Bi, keep_rows=max(1, Bo // 2), keep_cols=max(1, Bi // 2), dtype="bf16", seed=seed)
    blob = npas.pack_bb(dev(c.w, "bf16"), c.row_keep, c.col_keep, Bo, Bi)
    ydt = torch.bfloat16 if out_dtype is None else out_dtype
    r = (torch.randn(M, O, generator=torch.Generator().manual_seed(9))).to(ydt) if res else None
    ws = npas.workspace()
    kw = dict(relu=True, out_dtype=out_dtype, ws=ws, path=path, variant=variant)
    y = npas.linear_bb(dev(c.x, "bf16"), blob, dev(c.bias), None if r is None else r.cuda(), **kw)
    npas.check_device_status(ws)
    ref = oracle.linear_bb(c.x, c.w, c.row_keep, c.col_keep, Bo=Bo, Bi=Bi, bias=c.bias, relu=True,
                           residual=None if r is None else r.to(torch.float64).numpy())
    assert floored_rel_err(host(y), ref) < TOL_BF16
    assert torch.equal(y, npas.linear_bb(dev(c.x, "bf16"), blob, dev(c.bias), None if r is None else r.cuda(), **kw))


@pytest.mark.parametrize("bn,ks", [(16, 1), (16, 8), (32, 4), (64, 2), (64, 8), (128, 1), (128, 8)])
@pytest.mark.parametrize("M,I,O", [(1, 512, 256), (49, 2048, 128), (128, 192, 64), (129, 584, 72)])
def test_every_split_matches_oracle(M, I, O, bn, ks):
    """Splits with CTAs that have no steps (192 columns = three steps over eight CTAs), a second row tile of one row, a last
    column tile of eight columns, an input width that ends inside a step."""
    _run(M, I, O, 8, 8, variant=bn | (ks << 16), path=5, res=M != 1)


@pytest.mark.parametrize("out_dtype", [None, torch.float32])
@pytest.mark.parametrize("M,I,O,Bo", [(64, 2048, 1000, 40), (1, 1024, 1000, 8), (200, 584, 1000, 50)])
def test_classifier_widths_run_on_tensor_cores(M, I, O, Bo, out_dtype):
    _run(M, I, O, Bo, 8, out_dtype=out_dtype)


@pytest.mark.parametrize("out_dtype", [None, torch.float32])
@pytest.mark.parametrize("M,I,O", [(5000, 64, 1000), (300, 72, 24), (2000, 256, 264)])
def test_persistent_kernel_takes_ragged_widths(M, I, O, out_dtype):
    _run(M, I, O, 8, 8, path=5, out_dtype=out_dtype, res=True)


def test_split_that_does_not_fit_one_wave_is_declined():
    c = inputs.linear_case(M=4096, I=512, O=512, keep_rows=8, keep_cols=8, dtype="bf16", seed=902)
    blob = npas.pack_bb(dev(c.w, "bf16"), c.row_keep, c.col_keep, 64, 64)
    with pytest.raises(npas.NpasError) as e:
        npas.linear_bb(dev(c.x, "bf16"), blob, path=5, variant=64 | (8 << 16))
    assert e.value.code == 8


@pytest.mark.parametrize("M,I,O,Bo,Bi,kr,kc", [(1, 64, 64, 64, 64, 64, 64), (33, 1088, 48, 16, 64, 11, 37), (31, 520, 24, 8, 8, 5, 3),
                                               (65, 30, 21, 7, 5, 7, 5), (40, 1280, 100, 50, 64, 49, 1)])
def test_float64_kernel_edges(M, I, O, Bo, Bi, kr, kc):
    """fp32 layers: row tiles of 32 with remainders, inputs of more than one phase of columns, kept counts that neither the
    matrix step (8 rows x 4 columns) nor the group of warps divides, rows that are not 16-byte aligned."""
    c = inputs.linear_case(M=M, I=I, O=O, Bo=Bo, Bi=Bi, keep_rows=lambda a, b: max(0, kr - (a + b) % 2), keep_cols=kc, dtype="f32", w_sigma=0.3,
                           seed=903)
    blob = npas.pack_bb(dev(c.w), c.row_keep, c.col_keep, Bo, Bi)
    res = torch.randn(M, O, generator=torch.Generator().manual_seed(3))
    y = npas.linear_bb(dev(c.x), blob, dev(c.bias), res.cuda(), relu=True)
    ref = oracle.linear_bb(c.x, c.w, c.row_keep, c.col_keep, Bo=Bo, Bi=Bi, bias=c.bias, relu=True, residual=res.to(torch.float64).numpy())
    assert floored_rel_err(host(y), ref) < TOL_F32
    assert torch.equal(y, npas.linear_bb(dev(c.x), blob, dev(c.bias), res.cuda(), relu=True))

"""The float64 GEMM where its shape changes: rows of X per CTA (8 to 32), warps that only move X and Y, phases of 512 and of
256 columns, one group of warps and many, and the two kernels on either side of their rule."""
import numpy as np
import pytest
import torch

import oracle
import paper_2012_00596_b200 as npas
from paper_2012_00596_b200 import inputs
from util import TOL_F32, dev, floored_rel_err, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,I,O,Bo,Bi,kr,kc", [
    (1, 64, 64, 64, 64, 32, 32), (9, 128, 512, 64, 64, 64, 64), (25, 512, 512, 64, 64, 32, 32), (57, 128, 448, 64, 64, 48, 48),
    (392, 512, 512, 64, 64, 32, 32), (391, 64, 512, 64, 64, 1, 64), (51, 128, 1000, 8, 64, 4, 32), (104, 64, 1000, 40, 64, 20, 16),
    (33, 640, 120, 40, 64, 33, 33), (16, 1088, 64, 64, 64, 16, 16), (300, 256, 512, 32, 32, 16, 32), (160, 512, 512, 16, 64, 8, 32),
    (200, 64, 1000, 8, 64, 4, 32), (700, 64, 512, 16, 64, 8, 16), (7, 36, 20, 4, 6, 2, 3), (65, 30, 33, 11, 10, 5, 0),
])
@pytest.mark.parametrize("dtype,residual", [("f32", False), ("f32", True), ("bf16", False), ("bf16", True)])
def test_float64_gemm_at_the_edges(M, I, O, Bo, Bi, kr, kc, dtype, residual):
    c = inputs.linear_case(M=M, I=I, O=O, Bo=Bo, Bi=Bi, keep_rows=kr, keep_cols=kc, dtype=dtype, seed=1101)
    res = inputs.rng_for(1102).standard_normal((M, O), dtype=np.float32) if residual else None
    if res is not None and dtype == "bf16":
        res = inputs.bf16_representable(res)
    blob = npas.pack_bb(dev(c.w, dtype), c.row_keep, c.col_keep, Bo, Bi)
    ws = npas.workspace()
    y = npas.linear_bb(dev(c.x, dtype), blob, dev(c.bias), None if res is None else dev(res, dtype), relu=False, ws=ws, path=1)
    npas.check_device_status(ws)
    ref = oracle.linear_bb(c.x, c.w, c.row_keep, c.col_keep, Bo=Bo, Bi=Bi, bias=c.bias, residual=res, relu=False)
    # one rounding to float32 (2^-24), or to bf16 (2^-9 of the value), of a float64 sum
    assert floored_rel_err(host(y), ref) < (TOL_F32 if dtype == "f32" else 2.0 ** -8)

"""First layer by whole output rows: odd heights and row counts, the narrowest and widest rows, filter counts from one chunk to
the widest, work ranges that start inside an image, and the sizes beyond it that the other first-layer kernel keeps."""
import pytest
import torch

import oracle
import paper_2012_00596_b200 as npas
from paper_2012_00596_b200 import inputs
from util import TOL_BF16, dev, floored_rel_err, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,H,W,K", [(1, 1, 2, 16), (1, 2, 2, 64), (2, 3, 6, 48), (3, 7, 10, 128), (1, 9, 256, 32), (3, 14, 256, 128), (5, 13, 254, 112),
                                     (1, 7, 252, 16), (40, 23, 16, 64), (300, 5, 4, 16), (1, 8, 258, 64), (1, 6, 10, 144)])
def test_edges(N, H, W, K):
    c = inputs.conv_case(N=N, H=H, W=W, C=3, K=K, Mb=16, Nb=3, R=7, S=7, stride=2, pad=3, keep=lambda fb, cb: (49, 30, 1, 0)[fb % 4], dtype="bf16",
                         relu=True, seed=1201)
    blob = npas.pack_bp(dev(c.w, "bf16"), c.tap_mask, c.Mb, c.Nb)
    x, bias, ws = dev(c.x, "bf16"), dev(c.bias), npas.workspace()
    ref = oracle.conv2d_bp(c.x, c.w, c.tap_mask, Mb=c.Mb, Nb=c.Nb, stride=2, pad=3, bias=c.bias, relu=True)
    y = npas.conv2d_bp(x, blob, bias, None, stride=2, pad=3, relu=True, ws=ws)
    assert floored_rel_err(host(y), ref) < TOL_BF16
    assert floored_rel_err(host(npas.conv2d_bp(x, blob, bias, None, stride=2, pad=3, relu=True, out_dtype=torch.float32, ws=ws)), ref) < TOL_BF16
    pooled = npas.conv2d_bp_maxpool(x, blob, bias, stride=2, pad=3, relu=True, ws=ws)
    npas.check_device_status(ws)
    assert (host(pooled) == oracle.maxpool2d(host(y).astype("float64"), R=3, stride=2, pad=1)).all()

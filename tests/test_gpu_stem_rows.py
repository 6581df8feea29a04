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


@pytest.mark.parametrize("H,W,K", [(23, 16, 64), (14, 256, 128), (9, 250, 48)])
@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
def test_nothing_outside_the_window_counts(H, W, K, bad):
    """One infinite or undefined input value: outputs whose 7x7 window does not cover it keep their bits (its weight there is no
    zero of the layer's, it has none)."""
    c = inputs.conv_case(N=1, H=H, W=W, C=3, K=K, Mb=16, Nb=3, R=7, S=7, stride=2, pad=3, keep=49, dtype="bf16", seed=1202)
    blob = npas.pack_bp(dev(c.w, "bf16"), c.tap_mask, c.Mb, c.Nb)
    x0, bias, ws = dev(c.x, "bf16"), dev(c.bias), npas.workspace()
    conv = lambda x: npas.conv2d_bp(x, blob, bias, None, stride=2, pad=3, out_dtype=torch.float32, ws=ws)
    pool = lambda x: npas.conv2d_bp_maxpool(x, blob, bias, stride=2, pad=3, relu=True, ws=ws)
    y0, z0 = conv(x0), pool(x0)
    cols = sorted({0, 1, 2, 3, 4, 5, W // 2, W // 2 + 1, W - 4, W - 3, W - 2, W - 1})
    for h in (0, H // 2, H - 1):
        for w in cols:
            x = x0.clone()
            x[0, h, w, (h + w) % 3] = bad
            y, z = conv(x), pool(x)
            covers = lambda n, v: (2 * torch.arange(n, device="cuda") - v).abs() <= 3
            hit = covers(y.shape[1], h)[:, None] & covers(y.shape[2], w)[None, :]
            assert torch.equal(y[0][~hit], y0[0][~hit]), (h, w)
            assert not torch.isfinite(y[0][hit]).any(), (h, w)
            hp = torch.nn.functional.max_pool2d(hit[None, None].float(), 3, 2, 1)[0, 0].bool()
            assert torch.equal(z[0][~hp], z0[0][~hp]), (h, w)
    npas.check_device_status(ws)

"""Kept-pairs convolution on tiles of consecutive positions: tiles that span rows and several images, a short last tile, a last
round split by filters, and the geometries that fall back to tiles of whole rows."""
import pytest
import torch

import oracle
import paper_2012_00596_b200 as npas
from paper_2012_00596_b200 import inputs
from util import TOL_BF16, dev, floored_rel_err, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [
    dict(N=1, H=3, W=3, C=16, K=32, Mb=16, Nb=16),                               # less than a tile
    dict(N=9, H=5, W=7, C=32, K=128, Mb=16, Nb=16),                              # four images under a tile
    dict(N=40, H=2, W=2, C=32, K=128, Mb=32, Nb=16),                             # rows of too many images: tiles of whole rows
    dict(N=3, H=11, W=126, C=48, K=64, Mb=16, Nb=16),                            # widest rows
    dict(N=2, H=6, W=100, C=64, K=256, Mb=16, Nb=16, keep=9),                    # every tap: large weight slots
    dict(N=3, H=9, W=13, C=32, K=256, Mb=64, Nb=32, R=1, S=1, pad=0, keep=1),
    dict(N=3, H=12, W=10, C=64, K=48, Mb=16, Nb=16, R=3, S=5, pad=1),            # fifteen taps
    dict(N=64, H=13, W=13, C=32, K=512, Mb=16, Nb=16),                           # last round in four parts
    dict(N=64, H=15, W=15, C=32, K=512, Mb=32, Nb=32, keep=2),                   # last round in two parts
    dict(N=150, H=12, W=12, C=16, K=96, Mb=16, Nb=16, keep=2),                   # last round of unstaged columns
])
def test_tiles_of_consecutive_positions(kw):
    kw = dict(dict(keep=3, residual=True), **kw)
    c = inputs.conv_case(dtype="bf16", seed=1301, **kw)
    blob, ws = npas.pack_bp(dev(c.w, "bf16"), c.tap_mask, c.Mb, c.Nb), npas.workspace()
    ref = oracle.conv2d_bp(c.x, c.w, c.tap_mask, Mb=c.Mb, Nb=c.Nb, stride=1, pad=c.pad, bias=c.bias, residual=c.residual, relu=c.relu)
    for odt in (torch.bfloat16, torch.float32):
        f = lambda: npas.conv2d_bp(dev(c.x, "bf16"), blob, dev(c.bias), dev(c.residual, "f32" if odt == torch.float32 else "bf16"), stride=1,
                                   pad=c.pad, relu=c.relu, out_dtype=odt, ws=ws, path=8)
        y = f()
        npas.check_device_status(ws)
        assert floored_rel_err(host(y), ref) < TOL_BF16
        assert torch.equal(y, f())

"""Split form of the dense-image convolution (few output tiles, a cluster of CTAs per tile): channel and tap splits with
remainders, slabs of 64, 32 and 16 channels, image groups narrower and wider than the filter tile, strides, fp32 output."""
import pytest
import torch

import oracle
import paper_2012_00596_b200 as npas
from paper_2012_00596_b200 import inputs
from util import TOL_BF16, dev, floored_rel_err, host

pytestmark = pytest.mark.gpu


def _run(c, variant=0, path=0, out_dtype=None):
    blob = npas.pack_bp(dev(c.w, "bf16"), c.tap_mask, c.Mb, c.Nb)
    ws = npas.workspace()
    res = dev(c.residual, "bf16" if out_dtype is None else "f32")
    f = lambda: npas.conv2d_bp(dev(c.x, "bf16"), blob, dev(c.bias), res, stride=c.stride, pad=c.pad, relu=c.relu, out_dtype=out_dtype, ws=ws,
                               path=path, variant=variant)
    y = f()
    npas.check_device_status(ws)
    ref = oracle.conv2d_bp(c.x, c.w, c.tap_mask, Mb=c.Mb, Nb=c.Nb, stride=c.stride, pad=c.pad, bias=c.bias, residual=c.residual, relu=c.relu)
    assert floored_rel_err(host(y), ref) < TOL_BF16
    assert torch.equal(y, f())


@pytest.mark.parametrize("nt,kc,kt", [(64, 1, 1), (64, 4, 2), (64, 2, 1), (16, 2, 2), (32, 1, 3), (32, 4, 1), (128, 4, 2)])
@pytest.mark.parametrize("stride", [1, 2])
def test_every_split_of_wide_layers(nt, kc, kt, stride):
    _run(inputs.conv_case(N=1, H=13, W=15, C=256, K=128, Mb=16, Nb=8, keep=3, dtype="bf16", residual=True, stride=stride, seed=1101),
         nt | (kc << 16) | (kt << 24), 6)


@pytest.mark.parametrize("kw,variant", [
    (dict(N=2, H=9, W=11, C=96, K=176, Mb=16, Nb=8), 96 | (3 << 16) | (2 << 24)),                 # 32-channel slabs, groups of 16, ragged filter tile
    (dict(N=2, H=9, W=11, C=96, K=176, Mb=16, Nb=8, stride=2), 128 | (3 << 16) | (1 << 24)),
    (dict(N=1, H=7, W=7, C=48, K=96, Mb=8, Nb=4), 96 | (3 << 16) | (1 << 24)),                    # 16-channel slabs, groups of 32
    (dict(N=1, H=7, W=7, C=80, K=192, Mb=16, Nb=16), 64 | (5 << 16) | (1 << 24)),
    (dict(N=1, H=7, W=7, C=80, K=192, Mb=16, Nb=16), 128 | (2 << 16) | (3 << 24)),                # the second filter tile holds one group
    (dict(N=1, H=12, W=10, C=64, K=64, Mb=1, Nb=1, R=1, S=1, pad=0), 32 | (1 << 16) | (1 << 24)),
    (dict(N=1, H=30, W=126, C=32, K=16, Mb=16, Nb=16), 16 | (1 << 16) | (3 << 24)),               # widest image, one filter group
    (dict(N=1, H=8, W=9, C=128, K=64, Mb=16, Nb=8, R=3, S=5, pad=1), 64 | (2 << 16) | (4 << 24)), # fifteen taps in ranges of four
    (dict(N=1, H=9, W=9, C=64, K=64, Mb=16, Nb=8, R=1, S=1, pad=0, stride=2), 64 | (1 << 16) | (1 << 24)),   # strided without phases
])
def test_splits_at_the_edges(kw, variant):
    c = inputs.conv_case(keep=lambda fb, cb: (fb + 2 * cb) % (kw.get("R", 3) * kw.get("S", 3) + 1), dtype="bf16", residual=True, seed=1102, **kw)
    _run(c, variant, 6)
    _run(c, variant, 6, torch.float32)


@pytest.mark.parametrize("kw", [dict(N=1, H=14, W=14, C=256, K=256), dict(N=1, H=7, W=7, C=512, K=512), dict(N=1, H=14, W=14, C=512, K=512, stride=2),
                                dict(N=7, H=45, W=37, C=96, K=176, stride=2), dict(N=2, H=28, W=28, C=128, K=128), dict(N=3, H=5, W=5, C=16, K=48)])
def test_automatic_choice_on_few_tiles(kw):
    _run(inputs.conv_case(Mb=16, Nb=8, keep=3, dtype="bf16", residual=True, seed=1103, **kw))

"""Convolutions of channels and filters in multiples of 16 on CTA pairs: partial last channel block, items of several filter groups."""
import pytest
import torch

import paper_2012_00596_b200 as npas
from paper_2012_00596_b200 import inputs
from test_gpu_conv import oracle_case, run_case
from util import TOL_BF16, floored_rel_err, host

pytestmark = pytest.mark.gpu

WIDE = 1 << 24


SHAPES = {"32x1": 32 | (1 << 16), "64x1": 64 | (1 << 16), "96x2": 96 | (2 << 16), "128x2": 128 | (2 << 16), "192x1": 192 | (1 << 16)}


# takes: the shapes (filters per item x position tiles per CTA) that have to be taken; all others have to be refused
@pytest.mark.parametrize("takes,kw", [
    ("32x1", dict(N=2, H=14, W=14, C=16, K=16, Mb=16, Nb=8, keep=3)),             # a quarter of a channel block, half of an item's filters
    ("32x1 64x1 96x2 128x2 192x1", dict(N=3, H=13, W=17, C=80, K=176, Mb=16, Nb=16, keep=4)),     # groups of 16, the last item lacks some
    ("64x1 128x2", dict(N=2, H=20, W=11, C=112, K=96, Mb=32, Nb=16, keep=9)),     # groups of 32, three chunks in the last block
    ("32x1 64x1 96x2 128x2 192x1", dict(N=1, H=30, W=30, C=272, K=272, Mb=16, Nb=16, keep=lambda fb, cb: (fb + cb) % 4)),   # blocks without taps; 17 groups of 16
    ("64x1 128x2", dict(N=2, H=9, W=30, C=128, K=320, Mb=16, Nb=8, keep=2)),      # groups of 64
    ("128x2", dict(N=2, H=12, W=12, C=48, K=128, Mb=8, Nb=8, keep=5)),            # groups of 128 beside a partial channel block
    ("32x1 64x1", dict(N=5, H=7, W=7, C=144, K=48, Mb=16, Nb=16, keep=3)),        # several images per tile: too few tiles for two
    ("64x1", dict(N=3, H=15, W=13, C=32, K=32, Mb=16, Nb=16, keep=4, stride=2)),  # by phases
    ("32x1 64x1 192x1", dict(N=2, H=29, W=40, C=96, K=208, Mb=16, Nb=8, keep=9, stride=2)),       # by phases, partial block, 13 groups of 16
    ("32x1 64x1", dict(N=2, H=11, W=10, C=48, K=80, Mb=16, Nb=8, keep=1, R=1, S=1, pad=0)),       # one tap
    ("32x1 64x1", dict(N=1, H=9, W=12, C=80, K=48, Mb=16, Nb=8, keep=4, R=4, S=4, pad=1, stride=2)),      # 16 taps, strided without phases
    ("32x1 64x1 96x2 128x2", dict(N=40, H=28, W=28, C=80, K=112, Mb=16, Nb=16, keep=3)),          # more items than CTA pairs
])
@pytest.mark.parametrize("shape", [None, *SHAPES])
def test_wide_form_matches_oracle(takes, kw, shape):
    c = inputs.conv_case(dtype="bf16", residual=True, seed=310, **kw)
    variant = WIDE | (SHAPES[shape] if shape else 0)
    if shape and shape not in takes.split():
        with pytest.raises(npas.NpasError) as e:
            run_case(c, path=7, variant=variant)
        assert e.value.code == 8
        return
    y = run_case(c, path=7, variant=variant)
    assert torch.equal(y, run_case(c, path=7, variant=variant))                   # run-to-run determinism
    assert floored_rel_err(host(y), oracle_case(c)) < TOL_BF16


@pytest.mark.parametrize("kw", [
    dict(N=64, H=28, W=28, C=80, K=176, Mb=16, Nb=8, keep=3),
    dict(N=32, H=40, W=40, C=144, K=96, Mb=16, Nb=16, keep=9, stride=2),
    dict(N=32, H=28, W=28, C=128, K=320, Mb=16, Nb=8, keep=3),
])
@pytest.mark.parametrize("out_dtype", [None, torch.float32])
def test_wide_form_is_chosen_and_agrees_with_the_shared_memory_form(kw, out_dtype):
    c = inputs.conv_case(dtype="bf16", residual=True, seed=311, **kw)
    blob = npas.pack_bp(torch.from_numpy(c.w).cuda().to(torch.bfloat16), c.tap_mask, c.Mb, c.Nb)
    assert npas.conv2d_bp_kernel(c.x.shape, blob, stride=c.stride, pad=1, relu=c.relu, bias=True, residual=True) == 7
    got, other = host(run_case(c, out_dtype=out_dtype)), host(run_case(c, path=6, out_dtype=out_dtype))
    # the same products summed in fp32 in another order, and at most one rounding to bf16 (2^-8 of a value) of each
    assert floored_rel_err(got, other) < (TOL_BF16 if out_dtype is None else 1e-3)


@pytest.mark.parametrize("wide", [0, WIDE])
@pytest.mark.parametrize("kw", [
    dict(N=24, H=27, W=56, C=64, K=64, Mb=16, Nb=8, keep=3),                      # two tiles share a slab; the last row of an image's last tile is missing
    dict(N=43, H=13, W=56, C=64, K=64, Mb=16, Nb=8, keep=9),                      # seven tiles per image: a slab each
    dict(N=24, H=28, W=28, C=64, K=256, Mb=16, Nb=16, keep=3),                    # two sets of filters, a pair keeps one of them
    dict(N=26, H=28, W=28, C=64, K=384, Mb=16, Nb=8, keep=2),                     # three sets, which do not divide the pairs: nothing stays
    dict(N=75, H=14, W=14, C=256, K=128, Mb=16, Nb=8, keep=2),                    # weights that do not fit
])
def test_several_items_per_pair(kw, wide):
    c = inputs.conv_case(dtype="bf16", residual=True, seed=312, **kw)
    y = run_case(c, path=7, variant=wide)
    assert floored_rel_err(host(y), oracle_case(c)) < TOL_BF16
    assert torch.equal(y, run_case(c, path=7, variant=wide))

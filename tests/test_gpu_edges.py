"""Degenerate and extreme inputs: a layer with nothing kept, one-pixel images, one-row GEMMs, the largest
kernel the format allows, and sizes the calls must refuse."""
import numpy as np
import pytest
import torch

import oracle
import paper_2012_00596_b200 as npas
from paper_2012_00596_b200 import inputs
from util import TOL_BF16, TOL_F32, dev, floored_rel_err, host

pytestmark = pytest.mark.gpu


def _conv(c, path=0):
    dt = c.dtype
    blob = npas.pack_bp(dev(c.w, dt), c.tap_mask, c.Mb, c.Nb)
    ws = npas.workspace()
    y = npas.conv2d_bp(dev(c.x, dt), blob, dev(c.bias), dev(c.residual, dt), stride=c.stride, pad=c.pad, relu=c.relu, ws=ws, path=path)
    npas.check_device_status(ws)
    return y


def _conv_ref(c):
    return oracle.conv2d_bp(c.x, c.w, c.tap_mask, Mb=c.Mb, Nb=c.Nb, stride=c.stride, pad=c.pad, bias=c.bias,
                            residual=c.residual, relu=c.relu)


@pytest.mark.parametrize("path,Mb,Nb", [(1, 16, 16), (3, 16, 16), (6, 16, 16), (7, 16, 16), (8, 16, 16), (6, 1, 1)])
def test_layer_with_nothing_kept_is_bias_plus_residual(path, Mb, Nb):
    c = inputs.conv_case(N=2, H=14, W=14, C=64, K=128, Mb=Mb, Nb=Nb, keep=0, dtype="bf16", residual=True, relu=False, seed=801)
    assert not c.tap_mask.any()
    y = host(_conv(c, path))
    want = inputs.bf16_representable((c.bias[None, None, None, :].astype(np.float32) + c.residual).astype(np.float32))
    assert np.array_equal(y, want)                                   # one rounding of an exact fp32 sum
    assert floored_rel_err(y, _conv_ref(c)) < TOL_BF16


@pytest.mark.parametrize("H,W", [(1, 1), (2, 3), (1, 17)])
def test_images_smaller_than_the_kernel(H, W):
    """3x3, pad 1 on images of one or two pixels per side: most taps fall on padding."""
    for path, kw in ((0, dict(C=64, K=64, Mb=16, Nb=16)), (8, dict(C=64, K=64, Mb=16, Nb=16)), (1, dict(C=8, K=8, Mb=4, Nb=4))):
        c = inputs.conv_case(N=3, H=H, W=W, keep=5, dtype="bf16", residual=True, seed=802, **kw)
        assert floored_rel_err(host(_conv(c, path)), _conv_ref(c)) < TOL_BF16, (path, H, W)


def test_largest_kernel_the_format_allows():
    """R*S = 64 taps (8x8), every bit of the tap word in use; CUDA-core kernel, fp32."""
    c = inputs.conv_case(N=1, H=9, W=10, C=4, K=4, Mb=2, Nb=2, R=8, S=8, pad=3, keep=lambda fb, cb: 64 - 21 * (fb + cb), dtype="f32",
                         act="normal", w_sigma=0.2, seed=803)
    assert int(c.tap_mask[0, 0]) == 2 ** 64 - 1
    y = _conv(c)
    assert floored_rel_err(host(y), _conv_ref(c)) < TOL_F32
    blob = npas.pack_bp(dev(c.w), c.tap_mask, 2, 2)
    assert np.array_equal(blob.data.cpu().numpy(), oracle.pack_bp(c.w, c.tap_mask, 2, 2, "f32"))


@pytest.mark.parametrize("M", [1, 7, 129])
@pytest.mark.parametrize("path", [0, 1, 3, 5, 6])
def test_gemm_with_few_rows_and_empty_blocks(M, path):
    c = inputs.linear_case(M=M, I=128, O=256, Bo=64, Bi=64, keep_rows=lambda a, b: 0 if (a + b) % 2 else 20,
                           keep_cols=lambda a, b: 24, dtype="bf16", seed=804)
    x, w = dev(c.x, "bf16"), dev(c.w, "bf16")
    blob = npas.pack_bb(w, c.row_keep, c.col_keep, 64, 64)
    ws = npas.workspace()
    y = npas.linear_bb(x, blob, dev(c.bias), relu=True, ws=ws, path=path)
    npas.check_device_status(ws)
    ref = oracle.linear_bb(c.x, c.w, c.row_keep, c.col_keep, Bo=64, Bi=64, bias=c.bias, relu=True)
    assert floored_rel_err(host(y), ref) < TOL_BF16


def test_gemm_with_nothing_kept_is_the_bias():
    c = inputs.linear_case(M=130, I=128, O=128, Bo=64, Bi=64, keep_rows=0, keep_cols=0, dtype="bf16", relu=False, seed=805)
    blob = npas.pack_bb(dev(c.w, "bf16"), c.row_keep, c.col_keep, 64, 64)
    for path in (0, 1, 3, 5, 6):
        y = host(npas.linear_bb(dev(c.x, "bf16"), blob, dev(c.bias), relu=False, out_dtype=torch.float32, path=path))
        assert np.array_equal(y, np.broadcast_to(c.bias, y.shape)), path


def test_empty_and_oversized_problems_are_refused():
    c = inputs.conv_case(N=1, H=4, W=4, C=16, K=16, Mb=16, Nb=16, keep=3, dtype="bf16", seed=806)
    blob = npas.pack_bp(dev(c.w, "bf16"), c.tap_mask, 16, 16)
    x0 = torch.empty((0, 4, 4, 16), dtype=torch.bfloat16, device="cuda")
    with pytest.raises(npas.NpasError) as e:
        npas.conv2d_bp(x0, blob)                                      # empty batch
    assert e.value.code == 2
    with pytest.raises(npas.NpasError) as e:                          # image smaller than the kernel without padding
        npas.conv2d_bp(dev(c.x[:, :2, :2], "bf16"), blob, pad=0)
    assert e.value.code == 2
    # weight tensors beyond what 32-bit blob offsets address are refused by the size call
    import ctypes
    from paper_2012_00596_b200 import binding as B
    lib = npas.load()
    d = B.BpDesc(16384, 16384, 3, 3, 16, 16, B.BF16, B.BF16, 9)
    size = ctypes.c_size_t(0)
    tm = np.zeros(4, dtype=np.uint64)
    assert lib.npas_pack_bp_size(ctypes.byref(d), tm.ctypes.data_as(ctypes.c_void_p), ctypes.byref(size)) == 2


def _header(blob):
    return blob.data[:128].view(torch.int32).tolist()


@pytest.mark.parametrize("dtype,path,M", [("f32", 1, 70), ("bf16", 1, 70), ("bf16", 3, 70), ("f32", 1, 7000), ("bf16", 1, 7000)])
def test_gemm_ignores_list_entries_outside_their_block(dtype, path, M):
    """Row and column numbers of a damaged blob index shared memory: one outside its block counts for nothing."""
    c = inputs.linear_case(M=M, I=128, O=96, Bo=32, Bi=64, keep_rows=8, keep_cols=16, dtype=dtype, seed=811)
    blob = npas.pack_bb(dev(c.w, dtype), c.row_keep, c.col_keep, 32, 64)
    h, rk, ck = _header(blob), c.row_keep.copy(), c.col_keep.copy()
    off_rows, off_cols = h[11], h[12]
    drop = lambda m, i: np.uint64(int(m) & ~(1 << [t for t in range(64) if int(m) >> t & 1][i]))
    rows = blob.data[off_rows: off_rows + 6 * 32].view(6, 32)
    cols = blob.data[off_cols: off_cols + 6 * 64].view(6, 64)
    if path == 1:                                    # (the gather kernel's tiles hold the rows in place: it reads no row list)
        for b, i, v in ((0, 0, 32), (1, 7, 255), (5, 3, 200)):
            rows[b, i] = v
            rk.flat[b] = drop(c.row_keep.flat[b], i)
    for b, i, v in ((0, 0, 64), (2, 15, 255), (4, 9, 128)):
        cols[b, i] = v
        ck.flat[b] = drop(c.col_keep.flat[b], i)
    ws = npas.workspace()
    y = npas.linear_bb(dev(c.x, dtype), blob, dev(c.bias), relu=c.relu, ws=ws, path=path)
    npas.check_device_status(ws)
    ref = oracle.linear_bb(c.x, c.w, rk, ck, Bo=32, Bi=64, bias=c.bias, relu=c.relu)
    assert floored_rel_err(host(y), ref) < (TOL_F32 if dtype == "f32" else TOL_BF16)


@pytest.mark.parametrize("dtype,path", [("f32", 1), ("bf16", 1), ("bf16", 3)])
@pytest.mark.parametrize("Mb,Nb", [(16, 8), (16, 16)])
def test_conv_ignores_pairs_outside_the_layer(dtype, path, Mb, Nb):
    """Channel blocks and taps of a damaged blob: nothing is read or written outside, unpacking included."""
    c = inputs.conv_case(N=2, H=9, W=11, C=48, K=32, Mb=Mb, Nb=Nb, keep=3, dtype=dtype, seed=812)
    blob = npas.pack_bp(dev(c.w, dtype), c.tap_mask, Mb, Nb)
    h = _header(blob)
    nPairs, off = h[11], h[13]
    pairs = blob.data[off: off + 4 * nPairs].view(torch.int32)
    tm, w = c.tap_mask.copy(), c.w.copy()
    for j, (cb, tap) in ((1, (0xFFFF, 0)), (3 * 2 + 2, (48 // Nb, 8)), (nPairs - 1, (0, 9)), (3 * 4, (0, 0x7FFF))):
        old = int(pairs[j])
        kept = [t for t in range(9) if int(c.tap_mask.flat[j // 3]) >> t & 1]
        assert old >> 16 == kept[j % 3]
        fb, ob = divmod(j // 3, 48 // Nb)
        w[fb * Mb:(fb + 1) * Mb, kept[j % 3] // 3, kept[j % 3] % 3, ob * Nb:(ob + 1) * Nb] = 0
        pairs[j] = (tap << 16 | cb) - (1 << 32 if tap >= 0x8000 else 0)
    ws = npas.workspace()
    y = npas.conv2d_bp(dev(c.x, dtype), blob, dev(c.bias), relu=c.relu, ws=ws, path=path)
    npas.check_device_status(ws)
    if path == 1:
        ref = oracle.conv2d_bp(c.x, w, tm, Mb=Mb, Nb=Nb, bias=c.bias, relu=c.relu)
        assert floored_rel_err(host(y), ref) < (TOL_F32 if dtype == "f32" else TOL_BF16)
    assert torch.isfinite(y).all()
    _, masks = npas.unpack_bp(blob)
    assert (npas.mask_to_numpy(masks) < 1 << 9).all()


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("N,H,W,C,K,Mb,Nb,R,stride", [(4, 150, 151, 6, 40, 20, 6, 3, 1), (4, 161, 129, 8, 18, 9, 8, 3, 1), (1, 9, 9, 512, 16, 16, 16, 3, 1),
                                                      (2, 131, 133, 3, 32, 16, 3, 3, 1), (3, 60, 60, 36, 24, 12, 12, 5, 2), (1, 40, 41, 100, 16, 8, 4, 3, 1)])
def test_float64_convolution_at_its_edges(dtype, N, H, W, C, K, Mb, Nb, R, stride):
    """Sixteen filters per CTA with ragged filter blocks, more steps than are described at a time, every number of shares of the
    pairs, blocks of channels that are not whole steps; the same sums in float64 whatever the split."""
    c = inputs.conv_case(N=N, H=H, W=W, C=C, K=K, Mb=Mb, Nb=Nb, R=R, S=R, stride=stride, pad=1,
                         keep=(R * R if C in (3, 512) else lambda fb, cb: (5 * fb + 3 * cb) % (R * R + 1)), dtype=dtype, residual=True, seed=821)
    y = _conv(c, 1)
    assert floored_rel_err(host(y), _conv_ref(c)) < (TOL_F32 if dtype == "f32" else TOL_BF16)
    assert torch.equal(y, _conv(c, 1))


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("M,I,O,Bo,Bi", [(3001, 508, 508, 4, 4), (2100, 520, 96, 32, 40), (9999, 66, 33, 33, 33), (1200, 1600, 160, 5, 64), (10000, 21, 30, 3, 7),
                                         (4800, 320, 31, 31, 64), (2500, 128, 64, 1, 16)])
def test_float64_gemm_of_small_blocks_at_its_edges(dtype, M, I, O, Bo, Bi):
    """A warp per block: rows of blocks that do not divide the outputs per CTA, several phases of columns, ragged rows of X, odd
    widths that no wide copy starts on, empty and full blocks; and the widest block rows it takes against the first it does not."""
    c = inputs.linear_case(M=M, I=I, O=O, Bo=Bo, Bi=Bi, keep_rows=lambda a, b: (a * 29 + b * 13) % (Bo + 1), keep_cols=lambda a, b: (a * 7 + b * 23) % (Bi + 1),
                           dtype=dtype, seed=831)
    r = torch.randn(M, O, generator=torch.Generator().manual_seed(9)).to(torch.bfloat16)
    blob, ws = npas.pack_bb(dev(c.w, dtype), c.row_keep, c.col_keep, Bo, Bi), npas.workspace()
    run = lambda: npas.linear_bb(dev(c.x, dtype), blob, dev(c.bias), r.to(torch.float32 if dtype == "f32" else torch.bfloat16).cuda(), relu=c.relu, ws=ws, path=1)
    y = run()
    ref = oracle.linear_bb(c.x, c.w, c.row_keep, c.col_keep, Bo=Bo, Bi=Bi, bias=c.bias, residual=r.double().numpy(), relu=c.relu)
    assert floored_rel_err(host(y), ref) < (TOL_F32 if dtype == "f32" else TOL_BF16)
    assert torch.equal(y, run())


@pytest.mark.parametrize("path", [0, 1, 3, 6, 7, 8])
def test_conv_and_values_that_are_not_finite(path):
    """Infinities and NaNs: nothing outside an output's window counts on any path, and what only pruned weights would meet counts
    for nothing where kept pairs alone are multiplied."""
    c = inputs.conv_case(N=2, H=12, W=13, C=64, K=128, Mb=16, Nb=16, keep=lambda fb, cb: (0 if cb == 2 and fb < 7 else 1 + (fb + cb) % 8), dtype="bf16",
                         relu=False, seed=841)
    x = dev(c.x, "bf16")
    blob, ws = npas.pack_bp(dev(c.w, "bf16"), c.tap_mask, 16, 16), npas.workspace()
    run = lambda v: npas.conv2d_bp(v, blob, dev(c.bias), ws=ws, path=path, out_dtype=torch.float32)
    y0 = run(x)
    for h, w in ((0, 0), (5, 6), (11, 12)):
        for bad in (float("inf"), float("nan")):
            v = x.clone()
            v[1, h, w, 40] = bad                     # a channel that seven of the eight filter blocks have pruned at every tap
            y = run(v)
            near = ((torch.arange(12, device="cuda") - h).abs() <= 1)[:, None] & ((torch.arange(13, device="cuda") - w).abs() <= 1)[None, :]
            assert torch.equal(y[0], y0[0]) and torch.equal(y[1][~near], y0[1][~near])
            if path in (1, 3, 8):
                assert torch.equal(y[1][..., :112], y0[1][..., :112])
    npas.check_device_status(ws)


@pytest.mark.parametrize("path", [0, 1, 3, 5, 6])
def test_gemm_and_values_that_are_not_finite(path):
    c = inputs.linear_case(M=200, I=192, O=256, Bo=64, Bi=64, keep_rows=32, keep_cols=32, dtype="bf16", relu=False, seed=842)
    x = dev(c.x, "bf16")
    blob, ws = npas.pack_bb(dev(c.w, "bf16"), c.row_keep, c.col_keep, 64, 64), npas.workspace()
    run = lambda v: npas.linear_bb(v, blob, dev(c.bias), ws=ws, path=path, out_dtype=torch.float32)
    y0, others = run(x), torch.arange(200, device="cuda") != 130
    element = torch.from_numpy(oracle.bb_element_mask(c.row_keep, c.col_keep, 256, 192, 64, 64)).cuda().bool()
    for i in (0, 77, 191):
        for bad in (float("inf"), float("nan")):
            v = x.clone()
            v[130, i] = bad
            y = run(v)
            assert torch.equal(y[others], y0[others])
            if path == 1:
                assert torch.equal(y[130][~element[:, i]], y0[130][~element[:, i]])
    npas.check_device_status(ws)

"""Blobs written by the kernel just ahead of the call that reads them: the compute kernels may start while it runs, and must not
look at the blob before it is done.  Copies into the blob and packing, back to back with the call inside one captured graph,
where no host work hides the order; every kernel that has set-up before its wait."""
import ctypes

import pytest
import torch

import paper_2012_00596_b200 as npas
from paper_2012_00596_b200 import binding, inputs
from paper_2012_00596_b200.resnet50 import Resnet50Stack
from util import dev

pytestmark = pytest.mark.gpu

CONVS = {                                   # N, H, C, K, Mb, Nb, path, variant, kernel id
    "split": (1, 14, 256, 256, 16, 8, 0, 0, 6), "pairs": (8, 14, 256, 256, 16, 8, 7, 0, 7), "image": (8, 14, 256, 256, 16, 8, 6, 0, 6),
    "kept pairs": (8, 28, 128, 256, 16, 16, 8, 0, 8), "shared": (2, 14, 64, 64, 16, 8, 3, 0, 3), "float64": (2, 14, 64, 64, 16, 8, 1, 0, 1),
    "first layer": (2, 64, 3, 64, 16, 3, 5, 0, 5),
}
LINEARS = {"split": (64, 2048, 1024, 0, 0, 5), "single": (3136, 512, 512, 5, 0, 5), "pairs": (3136, 512, 512, 6, 0, 6), "float64": (64, 512, 512, 1, 0, 1)}


def _captured(f):
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        f()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        out = f()
    return g, out


def _written_just_ahead(call, blobs):
    """call(blob) on one buffer that a kernel fills with another blob's bytes right before: as on each blob by itself."""
    live = type(blobs[0])(torch.empty_like(blobs[0].data), blobs[0].desc)
    want = [call(b) for b in blobs]
    assert not torch.equal(want[0], want[1])
    srcs = [b.data.view(torch.int32) for b in blobs]

    def chain():
        out = []
        for i in range(12):
            torch.bitwise_xor(srcs[i % 2], 0, out=live.data.view(torch.int32))       # (a kernel, not a copy by the copy engine)
            out.append(call(live))
        return out

    g, out = _captured(chain)
    for _ in range(5):
        for o in out:
            o.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(o, want[i % 2]) for i, o in enumerate(out))


@pytest.mark.parametrize("name", list(CONVS))
def test_conv_after_a_copy_into_its_blob(name):
    N, H, C, K, Mb, Nb, path, variant, kid = CONVS[name]
    R, stride, pad = (7, 2, 3) if C == 3 else (3, 1, 1)
    blobs = []
    for seed in (1501, 1502):               # other weights and other tap sets, equally many: the same layout
        c = inputs.conv_case(N=N, H=H, W=H, C=C, K=K, Mb=Mb, Nb=Nb, R=R, S=R, stride=stride, pad=pad, keep=R * R if C == 3 else 3, dtype="bf16", seed=seed)
        blobs.append(npas.pack_bp(dev(c.w, "bf16"), c.tap_mask, Mb, Nb))
    x, ws = dev(c.x, "bf16"), npas.workspace()
    assert npas.conv2d_bp_kernel(x.shape, blobs[0], stride=stride, pad=pad, path=path, variant=variant) == kid
    _written_just_ahead(lambda b: npas.conv2d_bp(x, b, stride=stride, pad=pad, ws=ws, path=path, variant=variant), blobs)
    if C == 3:
        _written_just_ahead(lambda b: npas.conv2d_bp_maxpool(x, b, stride=stride, pad=pad, ws=ws), blobs)
    npas.check_device_status(ws)


@pytest.mark.parametrize("name", list(LINEARS))
def test_linear_after_a_copy_into_its_blob(name):
    M, I, O, path, variant, kid = LINEARS[name]
    blobs = []
    for seed in (1503, 1504):
        c = inputs.linear_case(M=M, I=I, O=O, Bo=64, Bi=64, keep_rows=32, keep_cols=32, dtype="bf16", seed=seed)
        blobs.append(npas.pack_bb(dev(c.w, "bf16"), c.row_keep, c.col_keep, 64, 64))
    x, ws = dev(c.x, "bf16"), npas.workspace()
    assert npas.linear_bb_kernel(M, blobs[0], path=path, variant=variant) == kid
    _written_just_ahead(lambda b: npas.linear_bb(x, b, ws=ws, path=path, variant=variant), blobs)
    npas.check_device_status(ws)


@pytest.mark.parametrize("Bo", [16, 64])                   # a warp per block; warps that share a block
def test_linear_f32_after_the_kernels_that_write_its_bias_and_residual(Bo):
    """Both are results of the library's own kernels just ahead, which let their successors start before they have written anything."""
    M, I, O = 1000, 512, 512
    c = inputs.linear_case(M=M, I=I, O=O, Bo=Bo, Bi=64, keep_rows=Bo // 2, keep_cols=32, dtype="f32", seed=1506)
    blob, ws = npas.pack_bb(dev(c.w), c.row_keep, c.col_keep, Bo, 64), npas.workspace()
    x, others, heads = dev(c.x), [dev(c.x[::-1]), dev(c.x) * 3], [dev(c.x[:1]), dev(c.x[1:2])]
    bias, res = torch.empty((1, O), device="cuda"), torch.empty((M, O), device="cuda")

    def call(i, b, r):
        npas.linear_bb(others[i], blob, out=r, ws=ws)
        npas.linear_bb(heads[i], blob, out=b, ws=ws)
        return npas.linear_bb(x, blob, b.view(O), r, ws=ws)

    want = []
    for i in range(2):
        b, r = torch.empty_like(bias), torch.empty_like(res)
        npas.linear_bb(others[i], blob, out=r, ws=ws)
        npas.linear_bb(heads[i], blob, out=b, ws=ws)
        torch.cuda.synchronize()
        want.append(npas.linear_bb(x, blob, b.view(O), r, ws=ws))
    assert not torch.equal(want[0], want[1])
    g, out = _captured(lambda: [call(i % 2, bias, res) for i in range(12)])
    for _ in range(5):
        for o in out:
            o.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(o, want[i % 2]) for i, o in enumerate(out))
    npas.check_device_status(ws)


@pytest.mark.parametrize("path,dtype", [(1, "f32"), (1, "bf16"), (6, "bf16"), (7, "bf16"), (8, "bf16"), (0, "bf16")])
def test_conv_after_the_kernels_that_write_its_input_and_residual(path, dtype):
    """A chain of convolutions in which each reads two results of the ones just ahead; path 0 is the split form here."""
    N, H, C = (1, 14, 256) if path == 0 else (2, 14, 64)
    c = inputs.conv_case(N=N, H=H, W=H, C=C, K=C, Mb=16, Nb=16, keep=3, dtype=dtype, seed=1507)
    blob, ws, xs = npas.pack_bp(dev(c.w, dtype), c.tap_mask, 16, 16), npas.workspace(), [dev(c.x, dtype), dev(c.x[:, ::-1], dtype)]
    bufs = [torch.empty_like(xs[0]) for _ in range(3)]

    def chain(wait):
        out = []
        for i in range(6):
            r = xs[i % 2]
            for j in range(3):                     # x -> a, (a, x) -> b, (b, a) -> c
                src, res = (r, None) if j == 0 else (bufs[j - 1], r if j == 1 else bufs[j - 2])
                npas.conv2d_bp(src, blob, None, res, relu=True, out=bufs[j], ws=ws, path=path)
                wait()
            out.append(npas.conv2d_bp(bufs[2], blob, None, bufs[1], relu=True, ws=ws, path=path))
            wait()
        return out

    want = chain(torch.cuda.synchronize)
    assert not torch.equal(want[0], want[1])
    g, out = _captured(lambda: chain(lambda: None))
    for _ in range(5):
        for o in (*out, *bufs):
            o.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(o, w) for o, w in zip(out, want))
    npas.check_device_status(ws)


def test_pack_then_convolve_in_one_graph():
    """The packers' two kernels and the convolution on what they write; the scan lets its successor start early."""
    lib = npas.load()
    c = inputs.conv_case(N=1, H=14, W=14, C=256, K=256, Mb=16, Nb=8, keep=3, dtype="bf16", seed=1505)
    x, ws, w = dev(c.x, "bf16"), npas.workspace(), dev(c.w, "bf16")
    weights = [w, w.flip(0).contiguous()]
    want = [npas.conv2d_bp(x, npas.pack_bp(v, c.tap_mask, 16, 8), ws=ws) for v in weights]
    blob = npas.pack_bp(w, c.tap_mask, 16, 8)
    mask = torch.from_numpy(c.tap_mask.view("int64")).cuda()
    live = torch.empty_like(w)

    def chain():
        out = []
        for i in range(8):
            torch.bitwise_xor(weights[i % 2].view(torch.int16), 0, out=live.view(torch.int16))
            code = lib.npas_internal_pack_bp(ctypes.byref(blob.desc), binding._p(live), binding._p(mask), binding._p(blob.data),
                                             ctypes.c_size_t(blob.data.numel()), binding._stream())
            assert code == 0
            out.append(npas.conv2d_bp(x, blob, ws=ws))
        return out

    g, out = _captured(chain)
    for _ in range(5):
        for o in out:
            o.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(o, want[i % 2]) for i, o in enumerate(out))
    npas.check_device_status(ws)


@pytest.mark.parametrize("N", [1, 4])
def test_stack_after_copies_into_its_blobs(N):
    """A forward pass fetches the weights of its later layers early; the blobs are written by the kernels just ahead of it."""
    layers = inputs.config4(H=64)
    net = Resnet50Stack(layers if isinstance(layers, list) else layers.layers)
    x = torch.randn((N, 64, 64, 3), generator=torch.Generator().manual_seed(5)).to(torch.bfloat16).cuda()
    want = net.forward(x).clone()
    first = [b.data.view(torch.int32) for b in net.blobs[:6]]
    keep = [t.clone() for t in first]

    def chain():
        for t in reversed(first):
            t.zero_()
        for t, k in zip(reversed(first), reversed(keep)):
            torch.bitwise_xor(k, 0, out=t)
        return net.forward(x)

    g, y = _captured(chain)
    for _ in range(20):
        y.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(y, want)

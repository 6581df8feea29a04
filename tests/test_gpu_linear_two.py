"""Two GEMMs in one kernel: both results against float64, at the edges of row tiles, weight rings and slot rings, and the
network that runs on it against its layers one by one."""
import ctypes

import pytest
import torch

import paper_2012_00596_b200 as npas
from paper_2012_00596_b200 import binding as B, inputs
from paper_2012_00596_b200.resnet50 import Resnet50Stack

pytestmark = pytest.mark.gpu


def _layer(g, O, I):
    w = (torch.randn((O, I), generator=g, device="cuda") * (2.0 / I) ** 0.5).to(torch.bfloat16)
    keep = [torch.randint(0, 2 ** 62, (O // 64, I // 64), generator=g, device="cuda") for _ in range(2)]
    blob = npas.pack_bb(w, keep[0], keep[1], 64, 64)
    return blob, npas.unpack_bb(blob)[0].double(), torch.randn((O,), generator=g, device="cuda")


def _close(got, ref):
    # one rounding to bf16 (2^-9 of the value); fp32 sums of up to 512 products are off by 512 * 2^-24 of their size at most
    err = (got.double() - ref).abs() / (ref.abs() + 1e-3 * ref.square().mean().sqrt())
    assert err.max().item() < 1e-2


@pytest.mark.parametrize("M", [1, 127, 129, 128 * 148, 128 * 300 + 77])
@pytest.mark.parametrize("K1,N1,N2,residual,relu", [(64, 256, 64, True, (1, 1)), (64, 256, 128, True, (1, 1)), (128, 512, 128, True, (1, 0)),
                                                    (128, 512, 256, True, (0, 1)), (64, 64, 64, False, (1, 1)), (192, 192, 192, False, (0, 0))])
def test_two_layers_in_one_launch(M, K1, N1, N2, residual, relu):
    lib = npas.load()
    g = torch.Generator(device="cuda").manual_seed(M + K1 + N1 + N2)
    x = torch.randn((M, K1), generator=g, device="cuda").relu_().to(torch.bfloat16)
    res = torch.randn((M, N1), generator=g, device="cuda").to(torch.bfloat16) if residual else None
    (b1, w1, c1), (b2, w2, c2) = _layer(g, N1, K1), _layer(g, N2, N1)
    y1 = torch.full((M, N1), float("nan"), dtype=torch.bfloat16, device="cuda")
    y2 = torch.full((M, N2), float("nan"), dtype=torch.bfloat16, device="cuda")
    a = B.LinearDesc(M, K1, N1, B.BF16, B.BF16, relu[0], 1, int(residual), 0, 0)
    b = B.LinearDesc(M, N1, N2, B.BF16, B.BF16, relu[1], 1, 0, 0, 0)
    assert bool(lib.npas_internal_linear_two_preferred(ctypes.byref(a), ctypes.byref(b))) == (K1 == 64)
    ws = npas.workspace()
    first = None
    for _ in range(2):
        assert lib.npas_internal_linear_two(ctypes.byref(a), ctypes.byref(b1.desc), ctypes.byref(b), ctypes.byref(b2.desc), B._p(x), B._p(b1.data), B._p(c1),
                                            B._p(res), B._p(y1), B._p(b2.data), B._p(c2), B._p(y2), B._p(ws), ctypes.c_size_t(ws.numel()), 0, B._stream()) == 0
        npas.check_device_status(ws)
        first = first if first is not None else (y1.clone(), y2.clone())
    assert torch.equal(first[0], y1) and torch.equal(first[1], y2)
    ref = x.double() @ w1.T + c1.double()
    if residual:
        ref += res.double()
    _close(y1, ref.relu_() if relu[0] else ref)
    ref = y1.double() @ w2.T + c2.double()
    _close(y2, ref.relu_() if relu[1] else ref)


def test_what_it_does_not_take_is_refused():
    lib = npas.load()
    ok = dict(M=40000, I=64, O=256, x_dtype=B.BF16, y_dtype=B.BF16, relu=1, has_bias=1, has_residual=0, path=0, variant=0)

    def preferred(a, b):
        return lib.npas_internal_linear_two_preferred(ctypes.byref(B.LinearDesc(*{**ok, **a}.values())), ctypes.byref(B.LinearDesc(*{**ok, "I": 256, "O": 64, **b}.values())))

    assert preferred({}, {})
    for a, b in (({"I": 96}, {}), ({}, {"O": 320}), ({}, {"O": 72}), ({"y_dtype": B.F32}, {}), ({}, {"has_residual": 1}), ({}, {"M": 39999}), ({"path": 5}, {}),
                 ({}, {"variant": 64}), ({"I": 512, "O": 2048}, {"I": 2048}), ({"I": 128, "O": 512}, {"I": 512}), ({}, {"I": 320})):
        assert not preferred(a, b)


@pytest.mark.parametrize("N,H", [(1, 64), (8, 224), (33, 160)])
def test_network_with_layers_taken_together(N, H):
    net = Resnet50Stack(inputs.config4(H=H))
    x = torch.randn((N, H, H, 3), generator=torch.Generator(device="cuda").manual_seed(7), device="cuda").to(torch.bfloat16)
    before = npas.launch_count()
    y = net.forward(x)
    together = npas.launch_count() - before
    before = npas.launch_count()
    one_by_one = net.forward(x, keep=True)[0]
    assert together < npas.launch_count() - before - 2
    net.check()
    # the same sums in the same order, layer by layer
    err = (y.double() - one_by_one.double()).norm() / one_by_one.double().norm()
    assert err.item() < 1e-2

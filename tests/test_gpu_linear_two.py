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
    # and bit by bit what the two layers give one after the other (the same products in the same order of columns, one rounding each)
    z1 = npas.linear_bb(x, b1, c1, res, relu=bool(relu[0]), path=5)
    assert torch.equal(y1, z1)
    assert torch.equal(y2, npas.linear_bb(z1, b2, c2, relu=bool(relu[1]), path=5))


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
    assert y.shape[0] == N
    diff, ref = (y.double() - one_by_one.double()).flatten(1), one_by_one.double().flatten(1)
    assert (diff.norm() / ref.norm()).item() < 1e-2
    assert (diff.norm(dim=1) / ref.norm(dim=1)).max().item() < 1e-2              # of every image, so that a few wrong rows are not diluted


def _graph_ms(f):
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        f()
    torch.cuda.synchronize()
    g, e = torch.cuda.CUDAGraph(), [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    with torch.cuda.graph(g, stream=s):
        f()

    def once(n=20):
        e[0].record()
        for _ in range(n):
            g.replay()
        e[1].record()
        torch.cuda.synchronize()
        return e[0].elapsed_time(e[1]) / n

    once(50)
    return min(once() for _ in range(7))


@pytest.mark.parametrize("N,H,most", [(1, 64, 1.05), (16, 224, 1.03), (64, 224, 1.02)])
def test_tuned_network_keeps_two_layers_in_one_launch(N, H, most):
    """A plan of its own for every layer does not cost the launches that two layers share (64 images: 1.028 times the untuned network's
    time without them): the tuner times those too, and the tuned network is not slower than the untuned one, `most` being what a layer
    alone and in the network may differ in, more for networks whose layers take three microseconds."""
    net = Resnet50Stack(inputs.config4(H=H))
    x = torch.randn((N, H, H, 3), generator=torch.Generator(device="cuda").manual_seed(8), device="cuda").to(torch.bfloat16)

    def launches():
        before = npas.launch_count()
        y = net.forward(x)
        return npas.launch_count() - before, y

    untuned, y0 = launches()
    ms0 = _graph_ms(lambda: net.forward(x))
    plans = net.tune(x, reps=20)
    pairs = {k: v for k, v in plans.plans.items() if k.startswith("two:")}
    assert len(pairs) == 2 and all(v[0] in (1, 2) for v in pairs.values())        # 64 -> 256 -> 64, and the stage's last layer with 256 -> 128
    tuned, y1 = launches()
    apart = [i for i in range(1, len(net.layers)) if net._follows(i) and net._routes(x)[3 * i - 1] == 1]
    assert tuned == untuned + len(apart)
    net.check()
    assert ((y0.double() - y1.double()).norm() / y0.double().norm()).item() < 1e-2
    ms1 = _graph_ms(lambda: net.forward(x))
    assert ms1 < most * ms0, (ms0, ms1, pairs)
    # saved, loaded, and with a layer on a plan of its own beside which no launch of two was measured
    net.plans = npas.PlanCache.from_json(plans.to_json())
    assert launches()[0] == tuned
    net.plans.plans = {k: v for k, v in plans.plans.items() if not k.startswith("two:")}
    assert launches()[0] > untuned

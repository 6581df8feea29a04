"""The whole network with shortcut projections on a second stream (few images): same bits as layer by layer, on several streams
and threads at once, and inside a captured graph."""
import threading

import pytest
import torch

from paper_2012_00596_b200 import inputs
from paper_2012_00596_b200.resnet50 import Resnet50Stack

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,H", [(1, 64), (1, 224), (3, 96)])
def test_projections_beside_the_block(N, H):
    layers = inputs.config4(H=H)
    net = Resnet50Stack(layers if isinstance(layers, list) else layers.layers)
    xs = [torch.randn((N, H, H, 3), generator=torch.Generator().manual_seed(i)).to(torch.bfloat16).cuda() for i in range(3)]
    want = [net.forward(x, keep=True)[0] for x in xs]
    torch.cuda.synchronize()
    bad = []

    def work(i):
        with torch.cuda.stream(torch.cuda.Stream()):
            for _ in range(10):
                if not torch.equal(net.forward(xs[i]), want[i]):
                    bad.append(i)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(3)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
    x = xs[0].clone()
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        net.forward(x)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        y = net.forward(x)
    for i in (1, 2, 0):
        x.copy_(xs[i])
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(y, want[i])

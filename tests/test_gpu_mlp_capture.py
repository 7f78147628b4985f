"""Forward passes of few and of many samples captured in a CUDA graph, behind a copy of the
inputs, behind each other and behind a training step: the replay's results are bitwise those of
the same calls made directly."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2403_04267_gb300 import surrogate as S, workloads as W


@pytest.mark.parametrize("B", [7, 255, 20000])
def test_captured_forward_passes(B):
    rng = np.random.default_rng(3)
    st = torch.cuda.Stream()
    f = torch.from_numpy(rng.uniform(-1, 1, (B, 5)).astype(np.float32)).cuda()
    t = torch.from_numpy(rng.uniform(-1, 1, (B, 66)).astype(np.float32)).cuda()
    x, y, z, w = torch.empty_like(f), torch.empty_like(t), torch.empty_like(t), torch.empty_like(t)
    net = S.MLP(B, stream=st)
    theta = W.mlp_init(8, gain=1.5).astype(np.float32)

    def calls():
        x.copy_(f)
        net.forward(x, out=y)
        net.forward(x, out=z)
        net.train_step(x, t, 1e-2)
        net.forward(x, out=w)

    torch.cuda.synchronize()
    net.set_params(theta)
    with torch.cuda.stream(st):
        calls()
    torch.cuda.synchronize()
    direct = [q.cpu().numpy().copy() for q in (y, z, w)]
    net.set_params(theta)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        calls()
    for q in (x, y, z, w):
        q.fill_(-3.0)
    torch.cuda.synchronize()
    net.set_params(theta)
    with torch.cuda.stream(st):
        g.replay()
    torch.cuda.synchronize()
    net.check()
    for a, b in zip(direct, (y, z, w)):
        assert np.array_equal(a, b.cpu().numpy())

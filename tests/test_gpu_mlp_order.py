"""A forward pass of few samples is launched to overlap the kernel before it in the stream: it
must still see what that kernel writes, whether its weights (a training step, set_params), its
inputs (a copy) or a buffer the kernel before still reads (its outputs).  Bitwise against the
same calls with the stream waited for in between."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2403_04267_gb300 import surrogate as S, workloads as W


def _run(wait, B):
    st = torch.cuda.Stream()
    rng = np.random.default_rng(9)
    X = torch.from_numpy(rng.uniform(-1, 1, (3675, 5)).astype(np.float32)).cuda()
    T = torch.from_numpy(rng.uniform(-1, 1, (3675, 66)).astype(np.float32)).cuda()
    fresh = [torch.from_numpy(rng.uniform(-1, 1, (B, 5)).astype(np.float32)).cuda() for _ in range(6)]
    nets = [S.MLP(3675, stream=st) for _ in range(2)]
    torch.cuda.synchronize()
    for k, n in enumerate(nets):
        n.set_params(W.mlp_init(40 + k, gain=1.5).astype(np.float32))
    out, y, x = [], torch.empty((B, 66), device="cuda"), torch.empty((B, 5), device="cuda")
    torch.cuda.synchronize()

    def done():
        if wait:
            st.synchronize()

    with torch.cuda.stream(st):
        for f in fresh:
            for n in nets:
                x.copy_(f)
                done()
                n.forward(x, out=y)               # inputs written just before
                done()
                out.append(y.clone())             # outputs read just after
                done()
                n.train_step(X, T, 1e-2)
                done()
                n.forward(x, out=y)               # weights written just before
                done()
                n.forward(f, out=y)               # and again over the same outputs
                done()
                out.append(y.clone())
    st.synchronize()
    return [t.cpu().numpy() for t in out] + [n.get_params() for n in nets]


@pytest.mark.parametrize("B", [1, 32, 255, 3675])
def test_overlapped_forward_passes_see_what_was_written_before(B):
    for a, b in zip(_run(False, B), _run(True, B)):
        assert np.array_equal(a, b)

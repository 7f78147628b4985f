"""Edges of the training pass's tiles (32 samples), of the weight gradients' batch splits
(64-wide slices, split from 256 samples on) and of the forward pass's two kernels."""
import numpy as np
import pytest

from oracle import mlp_oracle as M
from paper_2403_04267_gb300 import surrogate as S, workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _theta(seed):
    return W.mlp_init(seed, gain=1.5).astype(np.float32)


def _data(B, seed):
    rng = np.random.default_rng(seed)
    X = rng.uniform(-1, 1, (B, 5)).astype(np.float32)
    return X, (np.sin(X @ rng.normal(size=(5, 66))) * 0.7).astype(np.float32)


def test_small_batches_match_the_persistent_kernel():
    """A batch of 20000 takes the persistent kernel, fewer samples the 32-sample tiles: every
    row bitwise the same (the same operands, the same order of K)."""
    X, _ = _data(20000, 3)
    net = S.MLP(20000)
    net.set_params(_theta(21))
    Xd = torch.from_numpy(X).cuda()
    big = net.forward(Xd).cpu().numpy()
    for B in (1, 7, 31, 32, 33, 127, 255, 4864, 4865):
        y = net.forward(Xd[100:100 + B].contiguous()).cpu().numpy()
        assert np.array_equal(y, big[100:100 + B]), B


# the existing gradient test's bound (normwise 1e-2 per layer: BF16 roundings of activations
# and gradients, 2^-9 each, that FP32 accumulation moves by one unit now and then)
@pytest.mark.parametrize("B", [1, 8, 31, 33, 64, 255, 256, 257, 640])
def test_gradient_at_the_edges_matches_oracle(B):
    theta = _theta(22)
    X, T = _data(B, 4)
    net = S.MLP(700)
    net.set_params(theta)
    # a larger batch first: what it leaves beyond B must not count
    Xf, Tf = _data(700, 5)
    net.gradient(torch.from_numpy(Xf).cuda(), torch.from_numpy(Tf).cuda())
    loss, g = net.gradient(torch.from_numpy(X).cuda(), torch.from_numpy(T).cuda())
    L_ref, g_ref = M.backward(theta.astype(np.float64), X.astype(np.float64), T.astype(np.float64), bf16=True)
    # outputs normwise within 1e-3 (the forward test's bound), |Y| and |Y - T| of one order
    assert abs(loss - L_ref) <= 5e-3 * L_ref
    g = g.cpu().numpy().astype(np.float64)
    for (Wa, ba), (Wr, br) in zip(M.unpack(g), M.unpack(np.asarray(g_ref))):
        for a, r in ((Wa, Wr), (ba, br)):
            assert np.linalg.norm(a - r) <= 1e-2 * np.linalg.norm(r) + 1e-12

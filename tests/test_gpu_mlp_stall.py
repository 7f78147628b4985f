"""Failure detection of the surrogate's kernels: in a build whose operand copies stop after a
few slices the waits for the others run out (20 ms there), the kernels end with the error flag
set, having waited for their own copies and MMAs, and the GPU goes on: the same calls of the
ordinary build give the oracle's results in the same process."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import mlp_oracle as M
from paper_2403_04267_gb300 import build, salec, surrogate as S, workloads as W

# copies after which a tile gets no more: inside the second layer's eight slices of 128 rows,
# inside its second tile's four slices of 256 rows, inside a GEMM's ten
STALL = 6


@pytest.fixture(scope="module")
def stalled(tmp_path_factory):
    out = tmp_path_factory.mktemp("stall")
    jobs = []
    for src in ("mlp_kernels.cu", "mlp_train.cu", "mlp_api.cu"):
        obj = str(out / src.replace(".cu", ".o"))
        jobs.append((obj, subprocess.Popen([build.nvcc(), "-c", "-Xcompiler", "-fPIC", "-std=c++17", *build.ARCH, "-O3",
                                            f"-DSALEC_MLP_TEST_STALL={STALL}", "-o", obj, os.path.join(build.CSRC, src)])))
    assert all(p.wait() == 0 for _, p in jobs)
    so = str(out / "libstall.so")
    subprocess.check_call([build.nvcc(), "-shared", *build.ARCH, "-o", so, *[o for o, _ in jobs]])
    L, ref = C.CDLL(so), salec.load()
    for n in ("salec_mlp_bytes", "salec_mlp_create", "salec_mlp_set_params", "salec_mlp_forward", "salec_mlp_gradient",
              "salec_mlp_check", "salec_mlp_destroy", "salec_gemm_bf16"):
        getattr(L, n).argtypes, getattr(L, n).restype = getattr(ref, n).argtypes, getattr(ref, n).restype
    return L


class Net:
    def __init__(self, L, batch_max, theta):
        self.L, nb = L, C.c_size_t()
        assert L.salec_mlp_bytes(batch_max, C.byref(nb)) == salec.SALEC_OK
        self.buf = torch.empty(nb.value, dtype=torch.uint8, device="cuda")
        self.h = C.c_void_p()
        assert L.salec_mlp_create(batch_max, C.c_void_p(self.buf.data_ptr()), nb.value, None, C.byref(self.h)) == salec.SALEC_OK
        assert L.salec_mlp_set_params(self.h, theta.ctypes.data_as(C.c_void_p)) == salec.SALEC_OK
        assert L.salec_mlp_check(self.h) == salec.SALEC_OK

    def close(self):
        self.L.salec_mlp_destroy(self.h)


def _ptr(t):
    return C.c_void_p(t.data_ptr())


def test_waits_that_run_out_end_the_kernels_and_nothing_else(stalled):
    theta = W.mlp_init(31, gain=1.5).astype(np.float32)
    rng = np.random.default_rng(6)
    X = rng.uniform(-1, 1, (20000, 5)).astype(np.float32)
    T = rng.uniform(-1, 1, (20000, 66)).astype(np.float32)
    Xd, Td = torch.from_numpy(X).cuda(), torch.from_numpy(T).cuda()
    Y = torch.zeros((20000, 66), device="cuda")
    # the forward kernels of few and of many samples, a training pass (both its tensor-core
    # kernels: a batch of 9000 has nine slices a split)
    for B in (45, 20000):
        net = Net(stalled, B, theta)
        assert stalled.salec_mlp_forward(net.h, _ptr(Xd), B, _ptr(Y)) == salec.SALEC_OK
        assert stalled.salec_mlp_check(net.h) == salec.SALEC_ECUDA
        net.close()
    net = Net(stalled, 9000, theta)
    loss = C.c_double()
    assert stalled.salec_mlp_gradient(net.h, _ptr(Xd), _ptr(Td), 9000, None, C.byref(loss)) == salec.SALEC_ECUDA
    net.close()
    # the bare GEMM stores nothing for a tile whose operands did not come
    A = torch.randn((256, 640), device="cuda").bfloat16()
    Bm = torch.randn((192, 640), device="cuda").bfloat16()
    Cm = torch.full((256, 192), -7.0, device="cuda")
    torch.cuda.synchronize()
    assert stalled.salec_gemm_bf16(256, 192, 640, _ptr(A), 640, 1, _ptr(Bm), 640, 1, _ptr(Cm), 192, None) == salec.SALEC_OK
    torch.cuda.synchronize()
    assert bool((Cm == -7.0).all())
    # K within the slices that come: the same build computes it
    assert stalled.salec_gemm_bf16(256, 192, 384, _ptr(A), 640, 1, _ptr(Bm), 640, 1, _ptr(Cm), 192, None) == salec.SALEC_OK
    torch.cuda.synchronize()
    ref = A[:, :384].float() @ Bm[:, :384].float().T
    assert float((Cm - ref).norm()) <= 1e-4 * float(ref.norm())
    # and the ordinary build goes on as ever
    good = S.MLP(20000)
    good.set_params(theta)
    for B in (45, 20000):
        y = good.forward(Xd[:B].contiguous()).cpu().numpy()
        r = M.forward(theta.astype(np.float64), X[:200].astype(np.float64), bf16=True)
        r = r[0] if isinstance(r, tuple) else r
        n = min(B, 200)
        assert np.linalg.norm(y[:n] - r[:n]) <= 1e-3 * np.linalg.norm(r[:n])

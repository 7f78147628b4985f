"""Host programs over the package's CUDA headers, for tests that need no GPU: the source is
compiled with nvcc and its output returned."""
import os
import subprocess

from paper_2403_04267_gb300 import build

CSRC = build.CSRC


def run(src: str, tmp_path, *, macros=()) -> str:
    cu, exe = tmp_path / "t.cu", tmp_path / "t"
    cu.write_text(src)
    subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "-O1", "-Xcompiler", "-ffp-contract=off", "-Xcompiler", "-pthread",
                    *macros, "-I", CSRC, "-o", str(exe), str(cu)], check=True, capture_output=True, text=True, timeout=300)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-2000:]
    return r.stdout


def nvcc_missing() -> bool:
    try:
        build.nvcc()
    except RuntimeError:
        return True
    return not os.path.isdir(CSRC)

"""The library is compiled without switching any of the compiler's diagnostics off, and no
kernel carries both __launch_bounds__ and __maxnreg__, which nvcc takes for an error."""
import os
import re

from paper_2403_04267_gb300 import build


def test_no_diagnostic_is_switched_off(monkeypatch):
    cmds = []

    class Done:
        def wait(self):
            return 0

    monkeypatch.setattr(build.subprocess, "Popen", lambda cmd, *a, **k: cmds.append(cmd) or Done())
    monkeypatch.setattr(build.subprocess, "check_call", lambda cmd, *a, **k: cmds.append(cmd))
    monkeypatch.setattr(build.os, "replace", lambda a, b: None)
    build.build(force=True)
    assert len(cmds) == len(build.SOURCES) + 1
    for cmd in cmds:
        assert not [t for t in cmd if "suppress" in t or t in ("-w", "--disable-warnings")]


def test_no_kernel_has_both_register_qualifiers():
    kernels = 0
    for f in sorted(os.listdir(build.CSRC)):
        src = open(os.path.join(build.CSRC, f)).read()
        src = re.sub(r"//[^\n]*|/\*.*?\*/", "", src, flags=re.S)
        for chunk in src.split("__global__")[1:]:
            head = re.split(r"[{;]|\btemplate\b|\bSALEC_", chunk)[0]
            kernels += 1
            assert not ("__launch_bounds__" in head and "__maxnreg__" in head), (f, head)
    assert kernels > 20

"""The default step form by grid size (no gravity): in FP64 the phase kernels up to 256 x 256
cells and the fused form beyond, in the mixed form always the fused form; and in FP64 both
forms agree with each other at the repository's parity bar (1e-9 of a field's maximum) on grids of a few
cells, at the rule's edge and with fractions of several materials in a cell."""
import numpy as np
import pytest

from paper_2403_04267_gb300 import salec, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,small", [("fp64", "phases"), ("fp32mix", "fused")])
def test_default_form_by_size(precision, small):
    for nr, form in ((100, small), (256, small), (257, "fused")):
        s = salec.Sim(W.impact(nr, 256, 10.0, W.basalt(), None, 5, 9e3, 179, 16), precision=precision)
        assert s.step_form == form and s.launches_per_step() == (7 if form == "phases" else 3)
    s = salec.Sim(W.impact(40, 40, 10.0, W.basalt(), None, 3, 9e3, 28, 4, gravity=1.62), precision=precision)
    assert s.step_form == "phases"


@pytest.mark.parametrize("nr,nz,proj,strength", [(9, 13, False, False), (33, 17, True, True), (64, 50, True, False),
                                                 (257, 256, False, False)])
def test_forms_agree(nr, nz, proj, strength):
    spec = W.impact(nr, nz, 10.0, W.basalt(strength=strength), W.iron() if proj else None, 3, 9e3, int(0.7 * nz),
                    2 if nr < 20 else 6)
    a, b = salec.Sim(spec), salec.Sim(spec)
    a.step_form, b.step_form = "phases", "fused"
    for s in (a, b):
        s.step(40)
    names = ["f0", "rho0", "I", "vr", "vz", "pmax"] + (["f1", "rho1"] if proj else []) + \
            (["srr", "szz", "srz", "D"] if strength else [])
    for n in names:
        x, y = a.get(n), b.get(n)
        assert np.max(np.abs(x - y)) <= 1e-9 * max(np.max(np.abs(y)), 1e-300), n
    sa, sb = a.scalars(), b.scalars()
    assert sa["status"] == sb["status"] == 0 and abs(sa["t"] - sb["t"]) <= 1e-9 * sb["t"]

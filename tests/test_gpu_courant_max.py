"""The Courant step after fused steps and a change of the state: phase 0, alone or batched,
forms the maximum of the rates of the state it finds, whatever maximum a fused step or a
checkpoint image left.  A run whose matter is brought to rest takes the step a fresh run with
the same fields takes (Eq. 14 with the sound speed alone), not the shorter one of the state
that is gone."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2403_04267_gb300 import salec, workloads as W

FIELDS = ("f0", "rho0", "I", "vr", "vz")


@pytest.mark.parametrize("precision", ["fp64", "fp32mix"])
@pytest.mark.parametrize("route", ["host write", "image", "buffer"])
@pytest.mark.parametrize("nxt", ["phases", "batch", "persistent batch", "fused"])
def test_no_maximum_of_an_earlier_state_enters_the_step(precision, route, nxt):
    spec = W.impact(60, 50, 10.0, W.basalt(), None, 4, 20e3, 35, 0, pml_alpha=0.0)
    st = torch.cuda.Stream()
    a = salec.Sim(spec, precision=precision, stream=st)
    a.step_form = "fused"
    a.step(5)
    moving = a.scalars()["dt"]
    if route != "host write":
        image = a.get_state()
        a = salec.Sim(spec, precision=precision, stream=st)
        if route == "image":
            a.set_state(image)
        else:
            with torch.cuda.stream(st):
                a.state[:image.size].copy_(torch.from_numpy(image))
            a.state_changed()
    rest = {n: a.get(n) for n in FIELDS}
    for n in ("I", "vr", "vz"):
        rest[n] = np.zeros_like(rest[n])
        a.set(n, rest[n])
    b = salec.Sim(spec, precision=precision, stream=st)
    for n in FIELDS:
        b.set(n, rest[n])
    for s in (a, b):
        s.set_time(0.0, 1.0)             # a long step before: the Courant limit decides
        s.step_form = "fused" if nxt == "fused" else "phases"
        if "batch" in nxt:
            batch = salec.Batch([s], stream=st)
            batch.persistent = nxt != "batch"
            batch.step(1)
        else:
            s.step(1)
    da, db = a.scalars()["dt"], b.scalars()["dt"]
    assert da == db and da > 1.5 * moving

"""A batch on a stream of its own, of runs last stepped alone in the fused form at an odd
count: the copies that bring their fields home are queued on the runs' stream and the batch's
stream waits for them, so nothing has to be waited for in between and the fields are bitwise
those of a batch whose work all goes on one stream."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2403_04267_gb300 import salec, workloads as W

FIELDS = ("f0", "rho0", "I", "vr", "vz", "pmax")


def _advance(precision, own_stream, persistent):
    st = torch.cuda.Stream()
    sims = [salec.Sim(W.impact(400, 300 + 7 * k, 10.0, W.basalt(), None, 5, 9e3, 200, 8), precision=precision, stream=st)
            for k in range(2)]
    for s in sims:
        s.step_form = "fused"
        s.step(1)                     # the fields are in the second copy when the batch is made
    b = salec.Batch(sims, stream=torch.cuda.Stream() if own_stream else st)
    b.persistent = persistent
    b.step(2)
    for s in sims:
        s.step(21)                    # ... and when it steps again, with these steps still queued
    b.step(3)
    for s in sims:
        s.step(1)
    b.run(chunk=4, max_steps=4)
    return sims


@pytest.mark.parametrize("persistent", [False, True])
@pytest.mark.parametrize("precision", ["fp64", "fp32mix"])
def test_batch_waits_for_the_runs_own_stream(precision, persistent):
    for a, b in zip(_advance(precision, True, persistent), _advance(precision, False, persistent)):
        for n in FIELDS:
            assert np.array_equal(a.get(n), b.get(n)), n
        sa, sb = a.scalars(), b.scalars()
        assert sa["nstep"] == sb["nstep"] == 1 + 2 + 21 + 3 + 1 + 4
        assert sa["t"] == sb["t"] and sa["dt"] == sb["dt"] and sa["status"] == sb["status"] == 0

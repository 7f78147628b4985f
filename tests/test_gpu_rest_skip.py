"""Tiles at rest are copied once and then only tested: against a run whose tiles all go
through the tile kernel, bitwise the same fields, through host writes (resting vertices
written as -0, which the copy returns as +0), checkpoints at odd step counts and changes of
the rest-copy mode."""
import numpy as np
import pytest

from paper_2403_04267_gb300 import salec, workloads as W

pytestmark = pytest.mark.gpu

FIELDS = ("f0", "rho0", "I", "vr", "vz", "pmax")


def _same(a, b, names):
    for n in names:
        assert np.array_equal(a.get(n), b.get(n)), n
    sa, sb = a.scalars(), b.scalars()
    assert sa["t"] == sb["t"] and sa["dt"] == sb["dt"] and sa["nstep"] == sb["nstep"]


# one tile and a bit each way, tiles that divide the grid, ragged ones; with strength the
# stress fields are copied too; a non-uniform grid forms its rate cell by cell
@pytest.mark.parametrize("precision", ["fp64", "fp32mix"])
@pytest.mark.parametrize("nr,nz,kind", [(33, 17, "plain"), (192, 160, "plain"), (201, 131, "strength"),
                                        (161, 150, "stretched")])
def test_tiles_copied_once_match_tiles_always_computed(nr, nz, kind, precision):
    spec = W.impact(nr, nz, 10.0, W.basalt(strength=kind == "strength"), None, 3, 9e3, int(0.7 * nz), 0, pml_alpha=0.0)
    if kind == "stretched":
        spec["grid"]["dr"] = W.stretched_sizes(nr - 9, 10.0, 0, 9)
    names = FIELDS + (("srr", "szz", "srz", "D") if kind == "strength" else ())
    a, b = salec.Sim(spec, precision=precision), salec.Sim(spec, precision=precision)
    a.step_form = b.step_form = "fused"
    b.set_rest_copy(0)
    for s in (a, b):
        s.step(5)
        if nr > 100 and s is a:
            q, tiles = a.fused_queue()
            assert q < tiles          # some tiles are at rest
        for n in ("vr", "vz"):
            v = s.get(n)
            s.set(n, np.where(v == 0.0, -0.0, v))
        s.step(7)
    _same(a, b, names)
    image = a.get_state()
    a.step(20)
    c = salec.Sim(spec, precision=precision)
    c.step_form = "fused"
    c.set_state(image)
    c.step(20)
    b.step(20)
    _same(a, b, names)
    _same(c, b, names)
    a.set_rest_copy(0)
    a.step(3)
    a.set_rest_copy(2)
    a.step(4)
    a.set_rest_copy(1)
    a.step(17)
    b.step(24)
    _same(a, b, names)

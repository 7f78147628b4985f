"""Tiles at rest with two and three materials, full and cut cells, with and without strength:
copied once and then only tested, against a run whose tiles all go through the tile kernel,
bitwise the same fields, also across batched steps between fused ones (in place, so the copies
of the tiles at rest start anew)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2403_04267_gb300 import salec, workloads as W


def _spec(nm, strength):
    nr, nz = 200, 170
    spec = W.impact(nr, nz, 10.0, W.basalt(strength=strength), W.iron(), 3, 9e3, 120, 0, pml_alpha=0.0)
    if nm == 3:
        # a second layer from within a row of cells, the projectile the third material
        spec["materials"] = [W.basalt(strength=strength), W.granite(strength=strength), W.iron()]
        spec["layers"] = [dict(mat=0, zlo=0.0, zhi=604.0, rho=0.0, I0=0.0, vz=0.0),
                          dict(mat=1, zlo=604.0, zhi=1200.0, rho=0.0, I0=0.0, vz=0.0)]
        spec["projectile"]["mat"] = 2
    return spec


@pytest.mark.parametrize("precision", ["fp64", "fp32mix"])
@pytest.mark.parametrize("nm,strength", [(2, False), (2, True), (3, False), (3, True)])
def test_rest_tiles_of_several_materials_and_batched_steps_between(nm, strength, precision):
    spec = _spec(nm, strength)
    st = torch.cuda.Stream()
    names = [f"{k}{m}" for m in range(nm) for k in ("f", "rho")] + ["I", "vr", "vz", "pmax"]
    names += ["srr", "szz", "srz", "D"] if strength else []
    a, b = (salec.Sim(spec, precision=precision, stream=st) for _ in range(2))
    for s in (a, b):
        s.step_form = "fused"
    b.set_rest_copy(0)
    batches = [salec.Batch([s], stream=st) for s in (a, b)]

    def same():
        for n in names:
            assert np.array_equal(a.get(n), b.get(n)), n
        sa, sb = a.scalars(), b.scalars()
        assert sa["t"] == sb["t"] and sa["dt"] == sb["dt"] and sa["nstep"] == sb["nstep"] and sa["status"] == sb["status"] == 0

    for s in (a, b):
        s.step(9)
    q, tiles = a.fused_queue()
    assert 0 < q < tiles                 # some tiles are at rest
    same()
    for s, t in zip((a, b), batches):
        s.step(1)
        t.step(3)
        s.step(8)
    q, tiles = a.fused_queue()
    assert 0 < q < tiles
    same()

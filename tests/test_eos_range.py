"""The FP64 form's shortcuts at the ends of the FP64 range.  The Tillotson form takes 1/rho and
1/w0 from one division of their product, which overflows long before they do: its pressure and
squared sound speed against the formulas in decimal arithmetic, which has no such range.  A sound
speed beyond FP64 comes out infinite (the Courant step then reports the failure), not as the
floor.  A volume that overflowed gives an infinite fraction.

Tolerance: some thirty operations and exponentials of arguments up to 745, each within 2^-53 (times
the argument): 1e-13 of the sum of the terms' magnitudes, taken ten times."""
import math
from decimal import Decimal as D, getcontext

import pytest

import host_build
from paper_2403_04267_gb300 import workloads as W

SRC = r"""
#include <cmath>
#include <cstdio>
#include "salec_device.cuh"
int main()
{
    salec_material s = {};
    s.eos = SALEC_EOS_TILLOTSON;
FIELDS
    const salec::Mat m = salec::to_mat<double>(s);
    const double x[] = {VALUES};
    for (unsigned k = 0; k < sizeof x / sizeof x[0]; k += 2) {
        double p, c2;
        salec::eos_eval<double>(m, x[k], x[k + 1], p, c2);
        std::printf("%a %a\n", p, c2);
    }
    std::printf("%a %a\n", salec::div_by(INFINITY, 3.0, 1.0 / 3.0), salec::div_by(-INFINITY, 3.0, 1.0 / 3.0));
    std::printf("%a %a\n", salec::div_by(NAN, 3.0, 1.0 / 3.0), salec::div_by(1.7e308, 0.5, 2.0));
}
"""


def _number(t):
    return float(t) if t.lstrip("-") in ("inf", "nan") else float.fromhex(t)


def _tillotson(mat, rho_in, I):
    """p and c^2 with the sums of their terms' magnitudes."""
    getcontext().prec = 60
    k = {n: D(float(mat[n])) for n in ("rho0", "A", "B", "E0", "a", "b", "alpha", "beta", "Eiv", "Ecv")}
    I, rho_f = D(I), D("1e-12") * k["rho0"]
    rho = max(D(rho_in), rho_f)
    eta = rho / k["rho0"]
    mu, w0 = eta - 1, I / (k["E0"] * eta * eta) + 1
    d = k["b"] * I / (w0 * w0 * k["E0"] * eta * eta)

    def branch(Ea, Eb, x, expanded):
        dx = -k["rho0"] / (rho * rho)
        p = [k["a"] * rho * I, k["b"] * rho * I / w0 * Ea, k["A"] * mu * Eb * Ea]
        r = [k["a"] * I, (k["b"] * I / w0 + 2 * d * I) * Ea, k["A"] / k["rho0"] * Eb * Ea]
        if expanded:
            r += [-k["beta"] * dx * k["A"] * mu * Eb * Ea, -2 * k["alpha"] * x * dx * (p[1] + p[2])]
        else:
            p.append(k["B"] * mu * mu)
            r.append(2 * k["B"] * mu / k["rho0"])
        i = [rho * k["a"], rho * k["b"] / w0 * Ea, -rho * d * Ea]
        c = r + [sum(p) / (rho * rho) * t for t in i]
        size = sum(map(abs, r)) + sum(map(abs, p)) / (rho * rho) * sum(map(abs, i))
        return sum(p), sum(c), sum(map(abs, p)), size

    cold = branch(D(1), D(1), D(0), False)
    if rho >= k["rho0"] or I <= k["Eiv"]:
        v = cold
    else:
        x = k["rho0"] / rho - 1
        v = branch((-k["alpha"] * x * x).exp(), (-k["beta"] * x).exp(), x, True)
        if I < k["Ecv"]:
            w = (I - k["Eiv"]) / (k["Ecv"] - k["Eiv"])
            v = [(1 - w) * a + w * b for a, b in zip(cold, v)]
    p, c2, sp, sc = v
    if D(rho_in) < rho_f:
        p, sp = p * D(rho_in) / rho_f, sp * D(rho_in) / rho_f
    return p, max(c2, D("0.01") * k["A"] / k["rho0"]), sp, sc


@pytest.mark.skipif(host_build.nvcc_missing(), reason="no nvcc")
@pytest.mark.parametrize("mat", [W.basalt(), W.iron()], ids=["basalt", "iron"])
def test_tillotson_over_the_whole_range(tmp_path, mat):
    rhos = [mat["rho0"] * f for f in (1e-40, 1e-13, 1e-9, 1e-3, 0.4, 0.9999, 1.0, 1.05, 3.0, 1e3, 1e6, 1e60, 1e90, 1e105)]
    Is = [0.0, 1.0, 0.9 * mat["Eiv"], 1.1 * mat["Eiv"], 2 * mat["Ecv"], 1e9, 1e20, 1e60, 1e100, 1e150, 1e200, 1e250, 1e290,
          1e299, 1e304, 1.7e308]
    pts = [(r, i) for r in rhos for i in Is]
    fields = "\n".join(f"    s.{k} = {float(mat[k]).hex()};" for k in ("rho0", "A", "B", "E0", "a", "b", "alpha", "beta", "Eiv", "Ecv"))
    src = SRC.replace("FIELDS", fields).replace("VALUES", ",".join(v.hex() for q in pts for v in q))
    out = [[_number(t) for t in line.split()] for line in host_build.run(src, tmp_path).splitlines()]
    for (r, i), (p, c2) in zip(pts, out):
        tp, tc, sp, sc = _tillotson(mat, r, i)
        if sp < D("1e290"):
            assert math.isfinite(p) and abs(D(p) - tp) <= D("1e-12") * sp, (r, i, p, tp)
        if max(sc, sp) < D("1e290"):
            assert math.isfinite(c2) and abs(D(c2) - tc) <= D("1e-12") * sc, (r, i, c2, tc)
        else:
            # a term overflows on the way: infinite, or still the value
            assert c2 == math.inf or abs(D(c2) - tc) <= D("1e-12") * sc, (r, i, c2, tc)
    assert out[-2] == [math.inf, -math.inf]
    assert math.isnan(out[-1][0]) and out[-1][1] == math.inf


@pytest.mark.gpu
@pytest.mark.parametrize("form", ["phases", "fused"])
def test_an_overflowing_energy_stops_the_run(form):
    """A cell whose energy is about to overflow has an infinite sound speed: the Courant step
    falls to zero, below dt_min, and the status word says so (bit 4) at once."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_04267_gb300 import salec
    spec = W.impact(60, 50, 10.0, W.basalt(), W.iron(), 4, 9e3, 30, 6, gravity=1.62)
    spec["grid"]["dt_min"] = 1e-9
    s = salec.Sim(spec)
    s.step_form = form
    s.step(3)
    assert s.scalars()["status"] == 0
    e = s.get("I")
    e[20, 5] = 1.7e308
    s.set("I", e)
    s.step(1)
    assert s.scalars()["status"] & 4

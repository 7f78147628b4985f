"""div_by, the quotient by the cell volume with a stored reciprocal: exactly 1 for a full cell,
and never more than 0.5 + 2^-40 units in the last place from the true quotient (the remainder
correction squares the reciprocal's error of a few units), for the uniform grid's reciprocal
(1 / V rounded once) and the non-uniform one (a product of two rounded reciprocals, against a
volume that is a rounded product itself)."""
from fractions import Fraction
import math

import numpy as np
import pytest

import host_build

SRC = r"""
#include <cstdio>
#include "salec_device.cuh"
int main()
{
    double x[] = {VALUES};
    for (unsigned k = 0; k < sizeof x / sizeof x[0]; k += 3) std::printf("%a\n", salec::div_by(x[k], x[k + 1], x[k + 2]));
}
"""


def _cases():
    rng = np.random.default_rng(11)
    out = []
    for k in range(3000):
        # column area and row height of the workloads' range (cells of 0.1 m to 10 km, radii to 1000 km)
        A, h = float(10.0 ** rng.uniform(-3, 10)), float(10.0 ** rng.uniform(-1, 4))
        b = A * h
        y = 1.0 / b if k % 2 == 0 else (1.0 / A) * (1.0 / h)
        f = float((1.0, rng.uniform(0, 1), 10.0 ** rng.uniform(-6, 0), rng.uniform(1, 1.5))[k // 2 % 4])
        out.append((b if f == 1.0 else f * b, b, y))
    # numerators one unit from the volume, and zero
    for a, b, y in out[:40]:
        out += [(float(np.nextafter(b, 0.0)), b, y), (float(np.nextafter(b, np.inf)), b, y), (0.0, b, y)]
    return out


@pytest.mark.skipif(host_build.nvcc_missing(), reason="no nvcc")
def test_quotient_by_the_cell_volume(tmp_path):
    cases = _cases()
    got = host_build.run(SRC.replace("VALUES", ",".join(v.hex() for c in cases for v in c)), tmp_path).split()
    assert len(got) == len(cases)
    for (a, b, y), g in zip(cases, got):
        q = float.fromhex(g)
        true = Fraction(a) / Fraction(b)
        if a == b:
            assert q == 1.0
        elif a == 0.0:
            assert q == 0.0
        else:
            ulp = Fraction(math.ulp(float(true)))
            assert abs(Fraction(q) - true) <= ulp * (Fraction(1, 2) + Fraction(1, 2 ** 40)), (a, b, y)

"""The FP32 bounds by which the FP64 form decides whether a cell's Courant rate can raise the
running maximum: up_f32(x) is never below |x| and down_f32(x) never above x, at the ends of the
FP32 range, across a mantissa carry, for infinities and NaN; and inside the range neither is
further off than 2^-18 of its argument (a few units of the 20 mantissa bits it reads)."""
import math
import struct

import numpy as np
import pytest

import host_build

SRC = r"""
#include <cstdio>
#include "salec_device.cuh"
int main()
{
    double x[] = {VALUES};
    for (double v : x) std::printf("%a %a\n", (double)salec::up_f32(v), (double)salec::down_f32(v));
}
"""


def _values():
    edges = []
    for e in (-149, -127, -126, -125, -124, -1, 0, 1, 126, 127, 128):
        v = 2.0 ** e
        edges += [np.nextafter(v, 0.0), v, np.nextafter(v, np.inf), 1.5 * v]
    # all mantissa bits set (the carry into the exponent), and the constants around 2^-125, 2^127
    edges += [float(np.nextafter(2.0 ** k, 0.0)) for k in range(-130, 130, 13)]
    edges += [1.2e-38, 1.3e-38, 2.3e-38, 2.35e-38, 1.7e38, 1.71e38, 2.9e38, 3.0e38, 3.4e38, 3.5e38, 1e300, 5e-324, 0.0]
    rng = np.random.default_rng(5)
    vals = [float(v) for v in edges] + [float(v) for v in 10.0 ** rng.uniform(-45, 45, 400)]
    return [-v for v in vals] + vals + [math.inf, -math.inf, math.nan]


@pytest.mark.skipif(host_build.nvcc_missing(), reason="no nvcc")
def test_bounds_hold_over_the_whole_range(tmp_path):
    vals = _values()
    lits = ",".join("__builtin_inf()" if v == math.inf else "-__builtin_inf()" if v == -math.inf else "__builtin_nan(\"\")"
                    if math.isnan(v) else v.hex() for v in vals)
    out = host_build.run(SRC.replace("VALUES", lits), tmp_path).splitlines()
    assert len(out) == len(vals)
    lo, hi = 2.0 ** -125, 2.0 ** 127
    for v, line in zip(vals, out):
        up, down = (float.fromhex(t) if "inf" not in t else math.inf for t in line.split())
        if math.isnan(v):
            assert up == math.inf
            continue
        assert up >= abs(v) and up > 0.0, v
        if v >= 0.0:
            assert 0.0 <= down <= v, v
        else:
            assert down <= 0.0, v       # (rates are not negative)
        if lo <= abs(v) < hi:
            assert up <= abs(v) * (1 + 2.0 ** -18), v
            if v > 0:
                assert down >= v * (1 - 2.0 ** -18), v
        assert struct.unpack("f", struct.pack("f", up))[0] == up

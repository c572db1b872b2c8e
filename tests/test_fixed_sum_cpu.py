"""The warp sum in fixed point (fx_addend, fx_total of csrc/tdse_fixed.cuh), on
the CPU: the header is compiled here with g++ and a warp's 32 values are summed
as the kernel sums them, against exact rational arithmetic.

Bound: every value is held to half a unit 2^(e - 1079) of the largest exponent
field e (32 values: 16 units), the integers are added exactly and the result is
rounded once to 53 bits."""
import shutil
import struct
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from test_fixed_cpu import CSRC

DRIVER = r"""
#include <cstdio>
#include <cstring>
#include "tdse_fixed.cuh"
using namespace tdse_fx;
int main() {
  double v[32];
  while (fread(v, sizeof v, 1, stdin) == 1) {
    int e = 0;
    uint64_t u[32];
    memcpy(u, v, sizeof v);
    for (int i = 0; i < 32; ++i) { int f = (int)((u[i] >> 52) & 0x7ff); e = f > e ? f : e; }
    uint32_t p0 = 0, p1 = 0; int32_t p2 = 0;
    for (int i = 0; i < 32; ++i) {
      const int64_t X = fx_addend((uint32_t)(u[i] >> 32), (uint32_t)u[i], e);
      p0 += (uint32_t)X & 0xfffffu; p1 += (uint32_t)(X >> 20) & 0xfffffu; p2 += (int32_t)(X >> 40);
    }
    printf("%d %lld\n", e, (long long)fx_total(p0, p1, p2));
  }
}
"""


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("needs g++")
    d = tmp_path_factory.mktemp("fxsum")
    (d / "d.cpp").write_text(DRIVER)
    subprocess.run(["g++", "-O1", "-std=c++17", "-x", "c++", "-I", CSRC, str(d / "d.cpp"), "-o", str(d / "d")], check=True)
    return str(d / "d")


def _values(kind, rng):
    if kind == "equal":
        return np.full(32, rng.uniform(1, 2)) * 2.0 ** rng.integers(-50, 50)
    if kind == "largest":
        return np.full(32, np.nextafter(2.0, 0.0)) * rng.choice([-1.0, 1.0])
    if kind == "normal":
        return rng.standard_normal(32)
    if kind == "wide":
        return rng.standard_normal(32) * 10.0 ** rng.uniform(-40, 40, 32)
    if kind == "one":
        v = np.zeros(32)
        v[rng.integers(32)] = rng.standard_normal()
        return v
    v = rng.standard_normal(32)              # cancelling
    v[16:] = -v[:16] * (1 + 1e-15 * rng.standard_normal(16))
    return v


@pytest.mark.parametrize("kind", ["equal", "largest", "normal", "wide", "one", "cancel"])
def test_sum_of_32(driver, kind):
    rng = np.random.default_rng(5)
    cases = [_values(kind, rng) for _ in range(200)]
    out = subprocess.run([driver], input=b"".join(struct.pack("<32d", *c) for c in cases), capture_output=True, check=True)
    for c, line in zip(cases, out.stdout.decode().splitlines()):
        e, T = map(int, line.split())
        assert abs(T) < 2 ** 62 + 32
        exact = sum(Fraction(float(x)) for x in c)
        unit = Fraction(2) ** (e - 1079)
        assert abs(T * unit - exact) <= 16 * unit
        if kind in ("one", "largest"):       # exact operands: only the final rounding is left
            assert T * unit == exact

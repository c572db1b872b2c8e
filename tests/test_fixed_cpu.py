"""The fixed-point arithmetic of the FP64 stencil (csrc/tdse_fixed.cuh), on the
CPU: the header is compiled here with g++ and its conversions, products and
sums are compared with exact integer and rational arithmetic.

Bounds, from the representation (operands cut to 2^-60 of the block's largest
value 2^e, coefficients against 2^ec, V in units of 2^-57 of their product):
- a conversion is below its value by less than one unit 2^(e - 60), and exact
  for values down to 2^-7 of the block's largest;
- a sum of five products is off by less than half a unit of V (rounded once),
  a quarter unit for each dropped low product, and the operands' cuts times
  their coefficients;
- the result is V's nearest double."""
import os
import shutil
import struct
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1308_1856_gb300", "csrc")

DRIVER = r"""
#include <cstdio>
#include <cstring>
#include <string>
#include <iostream>
#include "tdse_fixed.cuh"
using namespace tdse_fx;
static uint64_t rd() { std::string s; std::cin >> s; return std::stoull(s, nullptr, 16); }
int main() {
  std::string c;
  while (std::cin >> c) {
    if (c == "conv") { uint64_t u = rd(), m = rd();
      printf("%lld\n", (long long)fx_from_words(u >> 32, (uint32_t)u, (uint32_t)m << 20)); }
    else if (c == "small") { uint64_t u = rd(), m = rd();
      printf("%lld\n", (long long)fx_from_small(u >> 32, (uint32_t)u, (int)m)); }
    else if (c == "bits") { long long V; int E; std::cin >> V >> E; printf("%llx\n", (unsigned long long)fx_to_bits(V, E)); }
    else if (c == "diag") { uint64_t u = rd(); int ec; std::cin >> ec; long long q = fx_encode_diag(u, ec);
      printf("%lld %d\n", (long long)fx_diag_value(q), fx_diag_shift(q)); }
    else if (c == "coef") { uint64_t u = rd(); int ec; std::cin >> ec; printf("%lld\n", (long long)fx_coef(u, ec)); }
    else if (c == "scale") { uint64_t u = rd(); double d; memcpy(&d, &u, 8); int ec = 0; int ok = fx_scale(d, ec);
      printf("%d %d\n", ok, ec); }
    else if (c == "fits") { uint64_t u = rd(); double d; memcpy(&d, &u, 8); int ec; std::cin >> ec;
      printf("%d\n", fx_diag_fits(d, ec) ? 1 : 0); }
    else if (c == "sum") { int n; std::cin >> n; int64_t hh = 0, mm = kHalf;
      for (int i = 0; i < n; ++i) { long long x, k; std::cin >> x >> k; fx_mac(fx_limbs(x), fx_limbs(k), hh, mm); }
      printf("%lld\n", (long long)fx_value(hh, mm)); }
    else if (c == "prod") { long long x, k; std::cin >> x >> k;
      printf("%lld\n", (long long)fx_coef_product(fx_limbs(x), fx_limbs(k))); }
  }
}
"""


def bits(x):
    return struct.unpack("<Q", struct.pack("<d", x))[0]


def dbl(b):
    return struct.unpack("<d", struct.pack("<Q", b))[0]


def field(x):
    return (bits(x) >> 52) & 0x7FF


@pytest.fixture(scope="module")
def fx(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("g++ not found")
    d = tmp_path_factory.mktemp("fx")
    (d / "m.cpp").write_text(DRIVER)
    subprocess.run([cxx, "-O2", "-std=c++17", "-x", "c++", "-I", CSRC, str(d / "m.cpp"), "-o", str(d / "m")], check=True)

    def run(lines):
        r = subprocess.run([str(d / "m")], input="\n".join(lines), capture_output=True, text=True, check=True)
        return r.stdout.split("\n")[:-1]
    return run


def _values(rng, n, spread):
    return [float(rng.standard_normal() * 2.0 ** -rng.integers(0, spread + 1)) for _ in range(n)]


def test_conversion(fx):
    rng = np.random.default_rng(1)
    cases = []
    for spread in (0, 6, 40, 80):
        for _ in range(50):
            v = _values(rng, 4, spread) + [0.0, -0.0]
            s = 2.0 ** int(rng.integers(-900, 900))
            cases.append([x * s for x in v])
    lines, want = [], []
    for v in cases:
        e = max(field(x) for x in v)
        for x in v:
            lines.append(f"conv {bits(x):x} {e:x}")
            want.append((x, e))
    for (x, e), got in zip(want, fx(lines)):
        X, u = int(got), Fraction(2) ** (e - 1082)
        err = abs(Fraction(x)) - abs(X) * u
        assert abs(X) < 2 ** 60 and 0 <= err < u, (x, X)
        assert X == 0 or (X > 0) == (x > 0)
        if abs(x) >= 2.0 ** -7 * dbl(e << 52):
            assert err == 0


def test_conversion_of_small_blocks(fx):
    """Subnormal values and zeros beside values near the bottom of FP64's range."""
    vals = [0.0, 5e-324, -1e-310, 2.0 ** -1022, -3e-305, 2.0 ** -960]
    for top in range(1, len(vals)):
        e = max(1, max(field(v) for v in vals[:top + 1]))
        out = fx([f"small {bits(v):x} {e:x}" for v in vals[:top + 1]])
        for v, got in zip(vals, out):
            u = Fraction(2) ** (e - 1082)
            err = abs(Fraction(v)) - abs(int(got)) * u
            assert 0 <= err < u and (int(got) == 0 or (int(got) > 0) == (v > 0))


def test_result_is_the_nearest_double(fx):
    rng = np.random.default_rng(2)
    V = [0, 1, -1, 3, 2 ** 53, 2 ** 53 + 1, 2 ** 54 - 1, -(2 ** 60) + 1, 2 ** 59 + 2 ** 5]
    V += [int(rng.integers(-2 ** 62, 2 ** 62) >> int(rng.integers(0, 60))) for _ in range(400)]
    E = [int(rng.integers(64, 2001)) for _ in V]
    for v, e, got in zip(V, E, fx([f"bits {v} {e}" for v, e in zip(V, E)])):
        r, x = dbl(int(got, 16)), Fraction(v) * Fraction(2) ** (e - 1079)
        assert abs(Fraction(r) - x) <= abs(x) * Fraction(1, 2 ** 53), (v, e)


@pytest.mark.parametrize("dr,stencil", [(0.05, 5), (0.1, 5), (0.2, 3), (0.3, 5), (1.7, 3), (1e-3, 5)])
def test_sums_against_exact_arithmetic(fx, dr, stencil):
    """H x at a point: five products against rational arithmetic, and at most
    the rounding of the same sum in FP64 over the whole sample (2-norm)."""
    h2 = dr * dr
    c0, c1, c2 = ((30 / (24 * h2), -16 / (24 * h2), 1 / (24 * h2)) if stencil == 5 else (1 / h2, -0.5 / h2, 0.0))
    ok, ec = map(int, fx([f"scale {bits(c0):x}"])[0].split())
    assert ok == 1 and 4 * c0 <= 2.0 ** ec < 8.01 * c0
    rng = np.random.default_rng([stencil, int(1000 * dr)])
    n = 300
    D = [c0 * float(1 + 0.3 * rng.standard_normal()) for _ in range(n)]
    a = [c0 * float(rng.uniform(-0.6, 0.6)) for _ in range(2 * n)]
    v = [_values(rng, 7, 6) for _ in range(n)]
    q = [tuple(map(int, s.split())) for s in fx([f"diag {bits(d):x} {ec}" for d in D])]
    k1, k2 = map(int, fx([f"coef {bits(c1):x} {ec}", f"coef {bits(c2):x} {ec}"]))
    ka = list(map(int, fx([f"coef {bits(x):x} {ec}" for x in a])))
    lines, es = [], []
    for i in range(n):
        e = max(field(x) for x in v[i])
        X = list(map(int, fx([f"conv {bits(x):x} {e:x}" for x in v[i]])))
        assert q[i][1] == 0
        lines.append(f"sum 5 {X[0] + X[1]} {k1} {X[2] + X[3]} {k2} {X[4]} {q[i][0]} {X[5]} {ka[2 * i]} {X[6]} {ka[2 * i + 1]}")
        es.append(e)
    F = Fraction
    s_fx = s_64 = 0.0
    for i, out in enumerate(fx(lines)):
        got = F(dbl(int(fx([f"bits {int(out)} {es[i] + ec}"])[0], 16)))
        x = [F(t) for t in v[i]]
        b, d = F(a[2 * i]), F(a[2 * i + 1])
        exact = F(D[i]) * x[4] + F(c1) * (x[0] + x[1]) + F(c2) * (x[2] + x[3]) + b * x[5] + d * x[6]
        top = F(2) ** (es[i] - 1022)                          # above every value of the block
        unit = F(2) ** -57 * top * F(2) ** ec
        cut = F(2) ** -60 * top * (abs(F(D[i])) + 2 * abs(F(c1)) + 2 * abs(F(c2)) + abs(b) + abs(d))
        table = 5 * F(2) ** -59 * F(2) ** ec * top            # the coefficients' own cuts
        assert abs(got - exact) <= unit * F(7, 4) + cut + table + abs(exact) * F(1, 2 ** 53)
        f64 = D[i] * v[i][4]
        for c, y in ((c1, v[i][0] + v[i][1]), (c2, v[i][2] + v[i][3]), (a[2 * i], v[i][5]), (a[2 * i + 1], v[i][6])):
            f64 = float(F(c) * F(y) + F(f64))                 # a fused multiply-add, rounded once
        s_fx += float((got - exact) / (top * F(c0))) ** 2
        s_64 += float((F(f64) - exact) / (top * F(c0))) ** 2
    assert s_fx <= s_64, (s_fx, s_64)


def test_extreme_sums_do_not_overflow(fx):
    X, K = 2 ** 60 - 1, 2 ** 61
    c0 = 1.0
    ec = int(fx([f"scale {bits(c0):x}"])[0].split()[1])
    k1, k2 = map(int, fx([f"coef {bits(-16 / 30 * c0):x} {ec}", f"coef {bits(c0 / 30):x} {ec}"]))
    for lo in (0x7FFFFFFF, 0x80000000, 0xFFFFFFFF, 0):
        for sx in (1, -1):
            x = sx * ((X >> 32 << 32) | lo)
            for k in (K, -K, (K >> 32 << 32) - (1 << 32) + lo):
                terms = [(2 * x, k1 * sx), (2 * x, k2), (x, k), (x, k), (x, k)]
                got = int(fx(["sum 5 " + " ".join(f"{p} {r}" for p, r in terms)])[0])
                exact = Fraction(sum(p * r for p, r in terms), 2 ** 64)
                assert abs(got - exact) <= Fraction(7, 4)


def test_diagonal_encoding(fx):
    """Entries of both signs from far below to far above c0; a double within a
    factor of two of c0 is held exactly, larger ones to 2^-54 of themselves."""
    c0 = 30 / 24 / 0.01
    ec = int(fx([f"scale {bits(c0):x}"])[0].split()[1])
    rng = np.random.default_rng(5)
    vals = [c0, 1.9 * c0, 0.6 * c0, -c0, 0.0, 1e-3 * c0, 3.9 * c0, 8.1 * c0, 1e4 * c0, -1e6 * c0, 5e-324]
    vals += [float(c0 * 10 ** rng.uniform(-3, 6)) for _ in range(200)]
    for d, out in zip(vals, fx([f"diag {bits(d):x} {ec}" for d in vals])):
        m, s = map(int, out.split())
        err = abs(Fraction(m) * Fraction(2) ** (ec + s - 61) - Fraction(d))
        assert m % 32 == 0 and 0 <= s < 32 and abs(m) <= 2 ** 61
        assert (s == 0) == (abs(d) < 2.0 ** ec)
        assert err <= max(Fraction(2) ** (ec - 57), abs(Fraction(d)) * Fraction(1, 2 ** 54))
        if 0.5 * c0 <= abs(d) < 2 * c0:
            assert err == 0
    assert fx([f"fits {bits(2.0 ** (ec + 29)):x} {ec}", f"fits {bits(2.0 ** (ec + 30)):x} {ec}",
               f"fits {bits(float('nan')):x} {ec}", f"fits {bits(float('inf')):x} {ec}"]) == ["1", "0", "0", "0"]
    assert [r.split()[0] for r in fx([f"scale {bits(x):x}" for x in (0.0, 1e-30, 1e30, float("inf"), float("nan"))])] == ["0"] * 5


def test_coefficient_product(fx):
    rng = np.random.default_rng(6)
    for _ in range(50):
        a, b = float(rng.uniform(0.5, 0.578)), float(rng.uniform(-1, 1))
        ka, X = int(fx([f"coef {bits(a):x} 0"])[0]), int(fx([f"conv {bits(b):x} {1022:x}"])[0])
        got = int(fx([f"prod {ka} {X}"])[0])
        exact = Fraction(ka) * X / 2 ** 60
        assert abs(got - exact) <= 6 and abs(got) < 2 ** 61

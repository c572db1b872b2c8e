"""The arithmetic of the fixed-point walker's sums (csrc/tdse_fixed.cuh, compiled
here with g++) at the ends of its ranges: the extreme sums of both gauges stay
inside 64 bits, a neighbour's coefficient is exact, and the differences of the
velocity gauge are brought to 58 bits without losing any that are there.  Also the
norm and its inverse from an approximate reciprocal square root."""
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
#include <iostream>
#include <string>
#include "tdse_fixed.cuh"
using namespace tdse_fx;
int main() {
  std::string c;
  while (std::cin >> c) {
    if (c == "sum") {   // n terms; those from m on are subtracted as one, as the velocity gauge's imaginary part does
      int n, m; std::cin >> n >> m;
      int64_t hh = 0, mm = kHalf >> kFineBits, ch = 0, cm = 0;
      for (int i = 0; i < n; ++i) {
        long long x, k; std::cin >> x >> k;
        if (i < m) fx_mac(fx_limbs(x), fx_limbs(k), hh, mm);
        else fx_mac(fx_limbs(x), fx_limbs(k), ch, cm);
      }
      printf("%lld\n", (long long)fx_value(hh - ch, mm - cm, kFineBits));
    } else if (c == "coef") { std::string s; std::cin >> s; uint64_t u = std::stoull(s, nullptr, 16); double d;
      memcpy(&d, &u, 8); FxStencilCoef q = fx_stencil_coef(d); printf("%lld %d\n", (long long)q.q, q.e);
    } else if (c == "norm") { std::string s, t; std::cin >> s >> t; uint64_t u = std::stoull(s, nullptr, 16),
      v = std::stoull(t, nullptr, 16); double d, y, n, i; memcpy(&d, &u, 8); memcpy(&y, &v, 8); fx_norm(d, y, n, i);
      memcpy(&u, &n, 8); memcpy(&v, &i, 8); printf("%llx %llx\n", (unsigned long long)u, (unsigned long long)v);
    } else if (c == "bring") { long long a, b; std::cin >> a >> b; int n = fx_lead(a, b);
      printf("%d %lld %lld\n", n, (long long)fx_bring(a, n), (long long)fx_bring(b, n)); }
  }
}
"""


@pytest.fixture(scope="module")
def fx(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("g++ not found")
    d = tmp_path_factory.mktemp("fxw")
    (d / "m.cpp").write_text(DRIVER)
    # overflow of a signed sum would abort
    subprocess.run([cxx, "-O2", "-std=c++17", "-ftrapv", "-x", "c++", "-I", CSRC, str(d / "m.cpp"), "-o", str(d / "m")],
                   check=True)

    def run(lines):
        r = subprocess.run([str(d / "m")], input="\n".join(lines), capture_output=True, text=True, check=True)
        return r.stdout.split("\n")[:-1]
    return run


# the largest operand and coefficient of every term: two neighbours' sums, the
# diagonal, the couplings (kappa <= 3^-1/2) and the velocity gauge's differences
KAPPA = int(2 ** 61 / 3 ** 0.5)
LENGTH = [(2 ** 61 - 2, 2 ** 59 - 1), (2 ** 61 - 2, 2 ** 59 - 1), (2 ** 60 - 1, 2 ** 61 - 32), (2 ** 60 - 1, KAPPA),
          (2 ** 60 - 1, KAPPA)]
VELOCITY = LENGTH + [(2 ** 58 - 1, KAPPA), (2 ** 58 - 1, KAPPA)]


@pytest.mark.parametrize("terms,split", [(LENGTH, 5), (VELOCITY, 3)])
def test_extreme_sums(fx, terms, split):
    lines, want = [], []
    for lo in (None, 0x7FFFFFFF, 0x80000000, 0xFFFFFFFF, 0):
        for sx in (1, -1):
            for sc in (1, -1):
                t = []
                for i, (x, k) in enumerate(terms):
                    if lo is not None:           # the low words at which the signed limbs are largest
                        x, k = (x >> 32 << 32) - 2 ** 32 + lo, (k >> 32 << 32) - 2 ** 32 + lo
                    t.append((sx * x, (1 if i < split else sc) * k))
                lines.append(f"sum {len(t)} {split} " + " ".join(f"{x} {k}" for x, k in t))
                want.append(Fraction(sum((1 if i < split else -1) * x * k for i, (x, k) in enumerate(t)), 2 ** 61))
    for got, w in zip(fx(lines), want):
        # half a unit, and two for each dropped low product
        assert abs(int(got) - w) <= 2 * len(terms) + Fraction(1, 2)
        assert abs(w) < 2 ** 62              # 7 2^56 at no extra bits, three more


def test_neighbour_coefficients_are_exact(fx):
    rng = np.random.default_rng(3)
    vals = [-16 / 24 / 0.05 ** 2, 1 / 24 / 0.05 ** 2, -0.5, 2.0 ** -60, -2.0 ** 60] + \
        [float(s * 10 ** rng.uniform(-15, 15)) for s in (1, -1) for _ in range(50)]
    out = fx([f"coef {struct.unpack('<Q', struct.pack('<d', v))[0]:x}" for v in vals])
    for v, o in zip(vals, out):
        q, e = map(int, o.split())
        assert 2 ** 58 <= abs(q) < 2 ** 59 and Fraction(q) * Fraction(2) ** (e - 61) == Fraction(v)


def test_differences_keep_their_bits(fx):
    rng = np.random.default_rng(4)
    cases = [(0, 0), (1, 0), (0, -1), (2 ** 61 - 1, -5), (-2 ** 61 + 1, 2 ** 61 - 1)]
    cases += [tuple(int(rng.integers(-2 ** 61, 2 ** 61)) >> int(rng.integers(0, 61)) for _ in range(2)) for _ in range(200)]
    for (a, b), o in zip(cases, fx([f"bring {a} {b}" for a, b in cases])):
        n, p, q = map(int, o.split())
        for v, w in ((a, p), (b, q)):
            assert abs(w) <= 2 ** 58 and abs(Fraction(v) * Fraction(2) ** n - w) < 1
            assert n < 0 or w == v << n
        if a or b:
            assert max(abs(p), abs(q)) >= 2 ** 57 - 1


def test_norm_and_inverse(fx):
    """From a reciprocal square root up to two units off: the norm within 0.51 of a unit in
    the last place, the inverse within 0.51 of the norm's inverse as it is rounded."""
    rng = np.random.default_rng(5)
    hx = lambda v: f"{struct.unpack('<Q', struct.pack('<d', v))[0]:x}"
    db = lambda h: struct.unpack("<d", struct.pack("<Q", int(h, 16)))[0]
    lines, vals = [], []
    for _ in range(2000):
        s2 = float(rng.uniform(1, 4) * 2.0 ** int(rng.integers(-920, 1022)))
        y = float(1.0 / np.sqrt(s2))
        for _ in range(abs(k := int(rng.integers(-2, 3)))):
            y = float(np.nextafter(y, np.inf if k > 0 else 0.0))
        lines.append(f"norm {hx(s2)} {hx(y)}")
        vals.append(s2)
    for s2, o in zip(vals, fx(lines)):
        n, i = map(db, o.split())
        # |n - sqrt| <= 0.51 ulp  <=>  (n -+ 0.51 ulp)^2 brackets s2
        u = Fraction(51, 100) * Fraction(float(np.spacing(n)))
        assert (Fraction(n) - u) ** 2 <= Fraction(s2) <= (Fraction(n) + u) ** 2
        v = Fraction(51, 100) * Fraction(float(np.spacing(i)))
        assert abs(Fraction(i) - 1 / Fraction(n)) <= v

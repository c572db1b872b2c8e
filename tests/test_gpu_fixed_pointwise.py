"""H x point by point.  The fixed-point walker (csrc/tdse_walk_fixed.cuh) rounds
against the largest value in a lane's reach, so the 2-norm of a state says
nothing of a small value beside a large one: the first radial points of a high
partial wave, a wave function inside a steep wall, scattered values of all
magnitudes.  At every point the error, against the oracle in long double, is held
to what FP64 may lose there: six roundings of at most half a unit in the last
place in either part of the sum, each of a partial sum no larger than the
point's own terms in modulus, S: sqrt(2) 6 2^-53 S < 9 2^-53 S."""
import numpy as np
import pytest

import oracle
from gpu_helpers import apply_h_gpu, grid_of, make

pytestmark = pytest.mark.gpu

TOL = 9 * 2.0 ** -53
LIGHT = 137.035999084


def _terms(g, E, x):
    """The sum of the moduli of a point's terms."""
    a = np.pad(np.abs(x), ((1, 1), (2, 2)))
    r, h = g.r(), g.h
    l = np.arange(g.L + 1)[:, None]
    c0, c1, c2 = (30 / 24, 16 / 24, 1 / 24) if g.stencil == 5 else (1.0, 0.5, 0.0)
    V = -g.Z / r if g.vtable is None else g.vtable
    D = c0 / h ** 2 + l * (l + 1) / (2 * r ** 2) + V
    if g.stencil == 5 and g.ghost:
        D[:, 0] -= c2 / h ** 2
    m = a[1:-1]
    S = np.abs(D) * m[:, 2:-2] + (c1 * (m[:, 1:-3] + m[:, 3:-1]) + c2 * (m[:, :-4] + m[:, 4:])) / h ** 2
    lo, hi = a[:-2], a[2:]
    kap = lambda n: np.where(n > 0, n / np.sqrt(np.maximum(4.0 * n * n - 1.0, 1.0)), 0.0)
    if g.gauge == 0:
        return S + np.abs(E * r) * (kap(l) * lo[:, 2:-2] + kap(l + 1) * hi[:, 2:-2])
    A = abs(E) / LIGHT
    d = (lambda b: (8 * (b[:, 1:-3] + b[:, 3:-1]) + b[:, :-4] + b[:, 4:]) / (12 * h)) if g.stencil == 5 else \
        (lambda b: (b[:, 1:-3] + b[:, 3:-1]) / (2 * h))
    return S + A * (kap(l) * (d(lo) + l / r * lo[:, 2:-2]) + kap(l + 1) * (d(hi) + (l + 1) / r * hi[:, 2:-2]))


def _worst(N, dr, L, st, x, E, gauge="length", **kw):
    g = grid_of(N, dr, L, st, gauge=1 if gauge == "velocity" else 0, **kw)
    t = make(N, dr, L, st, gauge=gauge, **kw)
    got = apply_h_gpu(t, E, x)
    t.close()
    want = oracle.apply_H(g, E, x, "fld")
    S = _terms(g, E, x)
    ok = S > 1e-280
    assert np.all(got[~ok] == want[~ok]) or np.max(np.abs(got[~ok] - want[~ok])) < 1e-290
    return float(np.max(np.abs(got - want)[ok] / S[ok]))


def _waves(N, dr, L, seed, real=False):
    """Bound shapes r^(l+1) e^(-r/a) and a packet in every partial wave."""
    rng = np.random.default_rng(seed)
    r = np.arange(1, N + 1) * dr
    x = np.zeros((L + 1, N), np.complex128)
    for l in range(L + 1):
        z = rng.standard_normal(5) + (0 if real else 1j) * rng.standard_normal(5)
        for c, a in zip(z, (1.0, 2.0, 4.0)):
            x[l] += c * 0.75 ** l * np.exp((l + 1) * np.log(r / (a * (l + 1))) - r / a + (l + 1))
        w, k = 0.02 * N * dr + 2.0, 0.8 * rng.uniform(0.5, 1.5)
        wave = np.cos(k * r) if real else np.exp(1j * k * r)
        x[l] += 0.2 * z[3] * 0.75 ** l * np.exp(-((r - 0.4 * N * dr) / w) ** 2) * wave
    return x / np.sqrt(dr * np.sum(np.abs(x) ** 2))


GRIDS = [(1203, 0.05, 63, 5), (701, 0.1, 127, 3), (601, 0.2, 24, 5)]


@pytest.mark.parametrize("gauge,E", [("length", -0.06), ("length", 0.0), ("velocity", 0.9 * LIGHT)])
@pytest.mark.parametrize("N,dr,L,st", GRIDS)
def test_waves(N, dr, L, st, gauge, E):
    for real in (False, True):
        assert _worst(N, dr, L, st, _waves(N, dr, L, 5, real), E, gauge) <= TOL


@pytest.mark.parametrize("gauge,E", [("length", 0.05), ("velocity", 0.3 * LIGHT)])
@pytest.mark.parametrize("N,dr,L,st", GRIDS)
def test_values_of_all_magnitudes(N, dr, L, st, gauge, E):
    rng = np.random.default_rng(N)
    for spread in (8, 60, 400):
        x = (rng.standard_normal((L + 1, N)) + 1j * rng.standard_normal((L + 1, N))) * \
            2.0 ** -rng.uniform(0, spread, (L + 1, N))
        assert _worst(N, dr, L, st, x, E, gauge) <= TOL, spread


@pytest.mark.parametrize("gauge,E", [("length", 0.05), ("velocity", 0.3 * LIGHT)])
@pytest.mark.parametrize("N,dr,L,st", GRIDS)
def test_one_populated_wave(N, dr, L, st, gauge, E):
    """Rows that hold nothing but the coupling, and single values."""
    x = _waves(N, dr, L, 6)
    x[1:] = 0
    assert _worst(N, dr, L, st, x, E, gauge) <= TOL
    x[:] = 0
    x[L // 2, ::29] = 1.0 - 0.5j
    assert _worst(N, dr, L, st, x, E, gauge) <= TOL


@pytest.mark.parametrize("wall", [1e4, 1e8, 1e10, 1e11, -1e9])
@pytest.mark.parametrize("gauge,E", [("length", 0.05), ("velocity", 0.3 * LIGHT)])
def test_steep_table_potential(wall, gauge, E):
    N, dr, L = 1000, 0.1, 6
    r = np.arange(1, N + 1) * dr
    v = np.where(r > 80.0, wall, -1.0 / r)
    x = np.zeros((L + 1, N), np.complex128)
    for l in range(L + 1):
        x[l] = (1 + 0.3j) * 0.6 ** l * np.where(r < 80.0, np.sin(np.pi * (l + 1) * r / 80.0), 0.0)
        x[l] += 1e-9 * np.exp(-((r - 80.0) / 0.5) ** 2)
    assert _worst(N, dr, L, 5, x, E, gauge, vtable=v) <= TOL
    assert _worst(N, dr, L, 3, x, E, gauge, vtable=v) <= TOL

"""The fixed-point stencil (csrc/tdse_walk_fixed.cuh) in the single-instance
kernels, at the sizes where its strips (60 columns, two a lane) and the warps'
shares end, against the oracle on random states: the operator to 1e-14 relative
L2, one step to 1e-12 (the bounds of every FP64 path).  Also: magnitudes near
FP64's limits, grids whose coefficients the fixed-point form cannot hold (the
FP64 fallback), and non-finite states."""
import numpy as np
import pytest

import oracle
import tdse_workloads as W
from gpu_helpers import apply_h_gpu, grid_of, make, rel_l2

pytestmark = pytest.mark.gpu

PULSE = oracle.Pulse(E0=0.0534, omega=0.057, ncycles=2)
SHAPES = [(1, 0), (2, 1), (59, 3), (60, 4), (61, 5), (119, 2), (121, 40), (601, 7), (1203, 65)]


@pytest.mark.parametrize("st", [3, 5])
@pytest.mark.parametrize("N,L", SHAPES)
def test_operator_at_strip_edges(N, L, st):
    x = W.random_state(N, L, seed=N + L)
    for ghost, dr in ((0, 0.1), (1, 0.2)):
        t = make(N, dr, L, st, ghost=ghost)
        for E in (0.0, -0.31):
            assert rel_l2(apply_h_gpu(t, E, x), oracle.apply_H(grid_of(N, dr, L, st, ghost=ghost), E, x)) <= 1e-14
        t.close()


def _explicit_dt(N, dr, L, st):
    return W.converging_dt(N, dr, L, 2, st, 0.06)


@pytest.mark.parametrize("method,order", [("taylor", 1), ("taylor", 5), ("rk4", 4), ("lanczos", 1), ("lanczos", 6)])
@pytest.mark.parametrize("N,L,st", [(59, 3, 5), (61, 5, 3), (121, 40, 5), (1203, 65, 5)])
def test_propagators(N, L, st, method, order):
    dr, ra = 0.1, 0.8 * N * 0.1
    dt = _explicit_dt(N, dr, L, st)
    x = W.random_state(N, L, seed=N)
    t = make(N, dr, L, st, pulse=PULSE, absorber_r=ra)
    t.set_small_grid_path("off")
    t.set_state(x)
    t.time = 40.0
    t.propagate(method, order, dt, 2)
    got = t.get_state()
    t.close()
    want, _ = oracle.propagate(grid_of(N, dr, L, st), x, method, order, dt, 2, t0=40.0, pulse=PULSE, mask=oracle.Mask(ra))
    assert rel_l2(got, want) <= 1e-12, rel_l2(got, want)


@pytest.mark.parametrize("tableau", ["euler", "classic", "merson", "fehlberg", "dormand_prince"])
@pytest.mark.parametrize("N,L,st", [(60, 4, 3), (601, 33, 5)])
def test_tableaus(N, L, st, tableau):
    dr = 0.1
    dt = _explicit_dt(N, dr, L, st)
    x = W.random_state(N, L, seed=N + 1)
    t = make(N, dr, L, st, pulse=PULSE)
    t.set_state(x)
    t.time = 40.0
    sig = t.propagate_rk(tableau, dt, 2)
    got = t.get_state()
    t.close()
    want, wsig = oracle.propagate_rk(grid_of(N, dr, L, st), x, tableau, dt, 2, t0=40.0, pulse=PULSE)
    assert rel_l2(got, want) <= 1e-12
    assert abs(sig - wsig) <= 1e-8 * abs(wsig)


@pytest.mark.parametrize("scale", [1e-300, 1e-140, 1e140, 1e290])
def test_operator_at_extreme_magnitudes(scale):
    """H is linear; results that fall below FP64's normal range may round there (an absolute bound)."""
    x = W.random_state(300, 6, seed=3)
    t = make(300, 0.1, 6, 5)
    got = apply_h_gpu(t, 0.05, x * scale)
    t.close()
    want = oracle.apply_H(grid_of(300, 0.1, 6, 5), 0.05, x)
    assert np.linalg.norm(got / scale - want) <= 1e-14 * np.linalg.norm(want)


@pytest.mark.parametrize("dr", [9e-10, 1e10])
def test_coefficients_outside_the_fixed_point_form(dr):
    x = W.random_state(130, 3, seed=9)
    t = make(130, dr, 3, 5)
    assert rel_l2(apply_h_gpu(t, 0.0, x), oracle.apply_H(grid_of(130, dr, 3, 5), 0.0, x)) <= 1e-14
    t.close()


def test_table_potential_with_a_huge_entry():
    v = -1.0 / W.radial_grid(300, 0.1)
    v[137] = 1e30
    x = W.random_state(300, 4, seed=3)
    t = make(300, 0.1, 4, 5, vtable=v)
    got = apply_h_gpu(t, 0.02, x)
    t.close()
    want = oracle.apply_H(grid_of(300, 0.1, 4, 5, vtable=v), 0.02, x)
    keep = np.arange(300) != 137
    assert rel_l2(got[:, keep], want[:, keep]) <= 1e-14 and rel_l2(got[:, ~keep], want[:, ~keep]) <= 1e-14


@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_nonfinite_values_spread_as_in_fp64(bad):
    x = W.random_state(400, 5, seed=4)
    x[2, 130] = bad
    t = make(400, 0.1, 5, 5)
    got = apply_h_gpu(t, 0.05, x)
    t.close()
    want = oracle.apply_H(grid_of(400, 0.1, 5, 5), 0.05, x)
    fin = np.isfinite(want.real) & np.isfinite(want.imag)
    assert np.array_equal(fin, np.isfinite(got.real) & np.isfinite(got.imag))
    assert rel_l2(got[fin], want[fin]) <= 1e-14

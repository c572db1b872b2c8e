"""The velocity gauge's fixed-point walk (csrc/tdse_walk_fixed.cuh: differences in
the ring, K l coefficients, negated limbs) at the sizes where its strips (60
columns), chunks and the warps' shares end, at magnitudes near FP64's limits and
with non-finite values, against the oracle on random states: the operator to 1e-13
relative L2 (its bound in this gauge), one step to 1e-12."""
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
    t = make(N, 0.1, L, st, gauge="velocity")
    for A in (0.0, -0.7, 40.0):
        assert rel_l2(apply_h_gpu(t, A, x), oracle.apply_H(grid_of(N, 0.1, L, st, gauge=1), A, x)) <= 1e-13
    t.close()


@pytest.mark.parametrize("method,order", [("taylor", 5), ("rk4", 4), ("lanczos", 6), ("merson", 0)])
@pytest.mark.parametrize("N,L,st", [(59, 3, 5), (61, 5, 3), (121, 40, 5), (1203, 65, 5)])
def test_steps(N, L, st, method, order):
    dt = W.converging_dt(N, 0.1, L, 2, st, 0.06)
    x = W.random_state(N, L, seed=N)
    g = grid_of(N, 0.1, L, st, gauge=1)
    t = make(N, 0.1, L, st, pulse=PULSE, absorber_r=0.08 * N, gauge="velocity")
    t.set_state(x)
    t.time = 40.0
    if order:
        t.propagate(method, order, dt, 2)
        want, _ = oracle.propagate(g, x, method, order, dt, 2, t0=40.0, pulse=PULSE, mask=oracle.Mask(0.08 * N))
    else:
        t.propagate_rk(method, dt, 2)
        want, _ = oracle.propagate_rk(g, x, method, dt, 2, t0=40.0, pulse=PULSE, mask=oracle.Mask(0.08 * N))
    got = t.get_state()
    t.close()
    assert rel_l2(got, want) <= 1e-12, rel_l2(got, want)


@pytest.mark.parametrize("scale", [1e-300, 1e-290, 1e-140, 1e140, 1e290])
def test_operator_at_extreme_magnitudes(scale):
    """H is linear; results that fall below FP64's normal range may round there (an absolute bound)."""
    x = W.random_state(300, 6, seed=3)
    t = make(300, 0.1, 6, 5, gauge="velocity")
    got = apply_h_gpu(t, 3.0, x * scale)
    t.close()
    want = oracle.apply_H(grid_of(300, 0.1, 6, 5, gauge=1), 3.0, x)
    assert np.linalg.norm(got / scale - want) <= 1e-13 * np.linalg.norm(want)


@pytest.mark.parametrize("bad", [np.inf, np.nan])
@pytest.mark.parametrize("st", [3, 5])
def test_nonfinite_values_spread_as_in_fp64(bad, st):
    x = W.random_state(400, 5, seed=4)
    x[2, 130] = bad
    t = make(400, 0.1, 5, st, gauge="velocity")
    got = apply_h_gpu(t, 0.5, x)
    t.close()
    want = oracle.apply_H(grid_of(400, 0.1, 5, st, gauge=1), 0.5, x)
    fin = np.isfinite(want.real) & np.isfinite(want.imag)
    assert np.array_equal(fin, np.isfinite(got.real) & np.isfinite(got.imag))
    assert rel_l2(got[fin], want[fin]) <= 1e-13


def test_a_potential_outside_the_form():
    v = -1.0 / W.radial_grid(300, 0.1)
    v[137] = 1e30
    x = W.random_state(300, 4, seed=3)
    t = make(300, 0.1, 4, 5, vtable=v, gauge="velocity")
    got = apply_h_gpu(t, 0.7, x)
    t.close()
    want = oracle.apply_H(grid_of(300, 0.1, 4, 5, vtable=v, gauge=1), 0.7, x)
    keep = np.arange(300) != 137
    assert rel_l2(got[:, keep], want[:, keep]) <= 1e-13 and rel_l2(got[:, ~keep], want[:, ~keep]) <= 1e-13


@pytest.mark.parametrize("st", [3, 5])
def test_batch_at_strip_and_chunk_edges(st):
    from paper_1308_1856_gb300 import Batch
    shapes = [(1, 0), (2, 1), (59, 3), (60, 4), (61, 5), (62, 33), (120, 31), (121, 40), (601, 7), (1203, 65)]
    specs = [dict(N=N, dr=0.1, lmax=L, krylov=min(8, N * (L + 1)), E0=0.05, omega=0.057, ncycles=2, gauge="velocity",
                  dt=W.converging_dt(N, 0.1, L, min(8, N * (L + 1)), st, 0.05)) for N, L in shapes]
    b = Batch(specs, stencil=st)
    for i, (N, L) in enumerate(shapes):
        b.set_state(i, W.random_state(N, L, seed=i))
        b.set_time(i, 30.0)
    b.propagate(1)
    for i, ((N, L), s) in enumerate(zip(shapes, specs)):
        g = oracle.Grid(N=N, h=0.1, L=L, stencil=st, gauge=1)
        want, _ = oracle.propagate(g, W.random_state(N, L, seed=i), "lanczos", s["krylov"], s["dt"], 1, t0=30.0,
                                   pulse=oracle.Pulse(E0=0.05, omega=0.057, ncycles=2))
        assert rel_l2(b.get_state(i), want) <= 1e-12, (N, L, rel_l2(b.get_state(i), want))
    b.close()

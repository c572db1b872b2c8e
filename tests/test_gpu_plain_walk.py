"""The FP64 kernels of a handle without the fixed-point copy of its diagonal
(given back at a failed allocation, TDSE_FAIL_ALLOC), at the sizes where their
segments of 32 columns end, in both gauges, against the oracle on random states:
the operator to 1e-14 relative L2 (velocity gauge: 1e-13, its terms round in
another order), one step to 1e-12 (the bounds of every FP64 path).  The one-launch
Lanczos path does not apply to such a handle."""
import numpy as np
import pytest

import oracle
import tdse_workloads as W
from gpu_helpers import apply_h_gpu, grid_of, make, rel_l2

pytestmark = pytest.mark.gpu

PULSE = oracle.Pulse(E0=0.0534, omega=0.057, ncycles=2)
SHAPES = [(1, 0, 5), (31, 3, 3), (33, 5, 5), (257, 40, 3), (601, 33, 5)]


@pytest.fixture
def plain(monkeypatch):
    def make_plain(N, L, st, gauge="length", ghost=0):
        monkeypatch.setenv("TDSE_FAIL_ALLOC", "work")
        t = make(N, 0.1, L, st, pulse=PULSE, gauge=gauge, ghost=ghost)
        t.set_small_grid_path("off")
        t.propagate("lanczos", 1, 1e-3, 0)        # the failing allocation
        return t
    return make_plain


@pytest.mark.parametrize("gauge", ["length", "velocity"])
@pytest.mark.parametrize("N,L,st", SHAPES)
def test_operator(plain, N, L, st, gauge):
    x = W.random_state(N, L, seed=N + L)
    for ghost in (0, 1) if gauge == "length" else (0,):
        t = plain(N, L, st, gauge, ghost)
        for E in (0.0, -0.31):
            want = oracle.apply_H(grid_of(N, 0.1, L, st, ghost=ghost, gauge=int(gauge == "velocity")), E, x)
            assert rel_l2(apply_h_gpu(t, E, x), want) <= (1e-14 if gauge == "length" else 1e-13)
        t.close()


@pytest.mark.parametrize("gauge", ["length", "velocity"])
@pytest.mark.parametrize("method,order", [("taylor", 1), ("taylor", 5), ("rk4", 4), ("lanczos", 1), ("lanczos", 6),
                                          ("merson", 0), ("dormand_prince", 0)])
@pytest.mark.parametrize("N,L,st", SHAPES[1:])
def test_steps(plain, N, L, st, method, order, gauge):
    dt = W.converging_dt(N, 0.1, L, 2, st, 0.06)
    x = W.random_state(N, L, seed=N)
    g = grid_of(N, 0.1, L, st, gauge=int(gauge == "velocity"))
    t = plain(N, L, st, gauge)
    t.set_persistent_path("force")
    t.set_state(x)
    t.time = 40.0
    if order:
        t.propagate(method, order, dt, 2)
        want, _ = oracle.propagate(g, x, method, order, dt, 2, t0=40.0, pulse=PULSE)
    else:
        t.propagate_rk(method, dt, 2)
        want, _ = oracle.propagate_rk(g, x, method, dt, 2, t0=40.0, pulse=PULSE)
    got = t.get_state()
    assert not t.persistent_path_used
    t.close()
    assert rel_l2(got, want) <= 1e-12, rel_l2(got, want)


@pytest.mark.parametrize("method,order", [("taylor", 4), ("rk4", 4), ("lanczos", 6)])
def test_imaginary_time(plain, method, order):
    N, L, st = 257, 4, 5
    dt = 0.4 / (2.7 / 0.1 ** 2 + L * (L + 1) / (2 * 0.1 ** 2))
    x = W.random_state(N, L, seed=2)
    t = plain(N, L, st)
    t.set_state(x)
    t.propagate_imag(method, order, dt, 2)
    want = oracle.propagate_imag(grid_of(N, 0.1, L, st), x, method, order, dt, 2)[0]
    assert rel_l2(t.get_state(), want) <= 1e-12
    t.close()

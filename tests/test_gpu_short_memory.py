"""A failed allocation (TDSE_FAIL_ALLOC): the handle gives the fixed-point copy
of its diagonal back and the call runs on in FP64, without reading the memory
it gave back.  Every propagator whose work vectors, or whose per-step
observables' scratch, are allocated at that moment, against the oracle: 1e-12
relative L2 after two steps, the bound of every FP64 path; the guard bands stay
intact (they also refill the freed memory's neighbourhood)."""
import numpy as np
import pytest

import oracle
import tdse_workloads as W
from gpu_helpers import apply_h_gpu, grid_of, make, rel_l2

pytestmark = pytest.mark.gpu

PULSE = oracle.Pulse(E0=0.0534, omega=0.057, ncycles=2)
N, DR, L, ST = 1203, 0.1, 65, 5


@pytest.fixture
def failing(monkeypatch):
    def make_failing(name, gauge="length"):
        monkeypatch.setenv("TDSE_FAIL_ALLOC", name)
        monkeypatch.setenv("TDSE_GUARD_BYTES", "4096")
        t = make(N, DR, L, ST, pulse=PULSE, gauge=gauge)
        t.set_small_grid_path("off")
        return t
    return make_failing


@pytest.mark.parametrize("gauge", ["length", "velocity"])
@pytest.mark.parametrize("name,record", [("work", False), ("dip_partials", True)])
@pytest.mark.parametrize("method,order", [("taylor", 5), ("rk4", 4), ("lanczos", 6)])
def test_real_time(failing, method, order, name, record, gauge):
    x = W.random_state(N, L, seed=7)
    dt = W.converging_dt(N, DR, L, 2, ST, 0.06)
    t = failing(name, gauge)
    t.set_state(x)
    t.time = 40.0
    if record:
        t.record_dipole(4)
    t.propagate(method, order, dt, 2)
    got = t.get_state()
    t.check_guards()
    t.close()
    g = grid_of(N, DR, L, ST, gauge=1 if gauge == "velocity" else 0)
    want, _ = oracle.propagate(g, x, method, order, dt, 2, t0=40.0, pulse=PULSE)
    assert rel_l2(got, want) <= 1e-12, rel_l2(got, want)


@pytest.mark.parametrize("method,order", [("taylor", 4), ("rk4", 4), ("lanczos", 8)])
def test_imaginary_time(failing, method, order):
    """Without the failure the same call runs in fixed point: 1e-12 between the
    two states, so 2e-12 between their squared norms n and, as the energy is
    -ln(n / n_before) / (2 dt), 1e-12 / dt between the energies."""
    dt = 0.4 / (2.7 / DR ** 2 + L * (L + 1) / (2 * DR ** 2))
    x = W.smooth_state(N, DR, L, seed=3)
    out = []
    for name in ("work", ""):
        t = failing(name)
        t.set_state(x)
        e = t.propagate_imag(method, order, dt, 3)
        out.append((t.get_state(), e))
        t.check_guards()
        t.close()
    assert rel_l2(out[0][0], out[1][0]) <= 1e-12
    assert abs(out[0][1] - out[1][1]) <= 1e-12 / dt


def test_runge_kutta_and_the_operator(failing):
    x = W.random_state(N, L, seed=8)
    dt = W.converging_dt(N, DR, L, 2, ST, 0.06)
    t = failing("work")
    t.set_state(x)
    t.time = 40.0
    t.propagate_rk("dormand_prince", dt, 2)
    want, _ = oracle.propagate_rk(grid_of(N, DR, L, ST), x, "dormand_prince", dt, 2, t0=40.0, pulse=PULSE)
    assert rel_l2(t.get_state(), want) <= 1e-12
    assert rel_l2(apply_h_gpu(t, 0.05, x), oracle.apply_H(grid_of(N, DR, L, ST), 0.05, x)) <= 1e-14
    t.close()


def test_an_allocation_the_handle_cannot_make_room_for(failing):
    from paper_1308_1856_gb300 import TDSEError
    with pytest.raises(TDSEError):
        failing("psi")

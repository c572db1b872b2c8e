"""What the FP64 Lanczos combination keeps exactly, the fixed-point one
(csrc/tdse_combine_fixed.cuh) keeps too: a real state in imaginary time stays real, and
a partial wave of subnormal values, which without a field no other one feeds, keeps its size."""
import numpy as np
import pytest

import oracle
import tdse_workloads as W
from gpu_helpers import grid_of, make

pytestmark = pytest.mark.gpu

N, DR, L = 517, 0.1, 5


@pytest.mark.parametrize("m", [1, 8, 9, 16])
def test_imaginary_time_keeps_a_real_state_real(m):
    x = np.abs(W.smooth_state(N, DR, L, seed=m)).astype(np.complex128)
    dt = 0.1 * m / (2.7 / DR ** 2 + L * (L + 1) / (2 * DR ** 2))
    t = make(N, DR, L, 5)
    t.set_state(x)
    t.propagate_imag("lanczos", m, dt, 3)
    got = t.get_state()
    t.close()
    assert np.linalg.norm(got.real) > 0 and not np.any(got.imag)
    from paper_1308_1856_gb300 import Batch
    b = Batch([dict(N=N, dr=DR, lmax=L, krylov=m, dt=dt, E0=0.0, omega=0.057, ncycles=2)], stencil=5)
    b.set_state(0, x)
    b.propagate_imag(3)
    got = b.get_state(0)
    b.close()
    assert np.linalg.norm(got.real) > 0 and not np.any(got.imag)


@pytest.mark.parametrize("m", [2, 5, 8])
def test_a_subnormal_wave_keeps_its_size(m):
    """To 1e-3 of the oracle's: the recurrence rounds the vectors to 2^-1074, 2.5e-12 of the
    wave, and multiplies what was rounded by its growth outside the Krylov vectors' span a
    step (the FP64 oracle is off by 1e-6 at m = 8)."""
    x = W.smooth_state(N, DR, L, seed=m)
    rng = np.random.default_rng(m)
    x[L] = 1e-312 * (1.0 + rng.uniform(size=N)) * np.exp(0.03j * np.arange(N))
    dt = W.converging_dt(N, DR, L, m, 5, 0.0)
    want, _ = oracle.propagate(grid_of(N, DR, L, 5), x, "lanczos", m, dt, 1, precision="fld")
    top = np.max(np.abs(want[L]))
    assert top > 1e-312
    t = make(N, DR, L, 5)
    t.set_small_grid_path("off")
    t.set_state(x)
    t.propagate("lanczos", m, dt, 1)
    got = t.get_state()
    t.close()
    assert np.max(np.abs(got[L] - want[L])) <= 1e-3 * top
    from paper_1308_1856_gb300 import Batch
    b = Batch([dict(N=N, dr=DR, lmax=L, krylov=m, dt=dt, E0=0.0, omega=0.057, ncycles=2)], stencil=5)
    b.set_state(0, x)
    b.propagate(1)
    got = b.get_state(0)
    b.close()
    assert np.max(np.abs(got[L] - want[L])) <= 1e-3 * top

"""What the FP64 Lanczos combination keeps exactly, the fixed-point one
(csrc/tdse_combine_fixed.cuh) keeps too: a real state in imaginary time stays real."""
import numpy as np
import pytest

import tdse_workloads as W
from gpu_helpers import make

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

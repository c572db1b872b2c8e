"""The Lanczos combination in fixed point (csrc/tdse_combine_fixed.cuh) at the
sizes where its groups of eight vectors end, in the single-instance kernels, the
one-launch path and the batch, against the oracle after one converging step
(1e-12 relative L2, the per-step bound of every FP64 path); and states near FP64's
limits, whose warps take the FP64 sums."""
import numpy as np
import pytest

import oracle
import tdse_workloads as W
from gpu_helpers import grid_of, make, rel_l2

pytestmark = pytest.mark.gpu

PULSE = oracle.Pulse(E0=0.0534, omega=0.057, ncycles=2)
N, DR, L, ST = 517, 0.1, 9, 5


def _single(x, m, dt, path):
    t = make(N, DR, L, ST, pulse=PULSE, absorber_r=40.0)
    t.set_small_grid_path("off")
    t.set_persistent_path(path)
    t.set_state(x)
    t.time = 40.0
    t.propagate("lanczos", m, dt, 1)
    got = t.get_state()
    t.close()
    return got


def _want(x, m, dt):
    return oracle.propagate(grid_of(N, DR, L, ST), x, "lanczos", m, dt, 1, t0=40.0, pulse=PULSE, mask=oracle.Mask(40.0))[0]


@pytest.mark.parametrize("m", [1, 2, 7, 8, 9, 15, 16, 17, 24, 25, 32])
def test_group_edges(m):
    dt = W.converging_dt(N, DR, L, min(m, 16), ST, 0.06)
    x = W.random_state(N, L, seed=m)
    got = _single(x, m, dt, "off")
    assert rel_l2(got, _want(x, m, dt)) <= 1e-12
    assert np.array_equal(got, _single(x, m, dt, "force"))
    from paper_1308_1856_gb300 import Batch
    s = dict(N=N, dr=DR, lmax=L, krylov=m, dt=dt, E0=PULSE.E0, omega=PULSE.omega, ncycles=PULSE.ncycles, absorber_r=40.0)
    b = Batch([s], stencil=ST)
    b.set_state(0, x)
    b.set_time(0, 40.0)
    b.propagate(1)
    assert rel_l2(b.get_state(0), _want(x, m, dt)) <= 1e-12
    b.close()


@pytest.mark.parametrize("scale", [1e-300, 1e-270, 1e-140, 1e140])
def test_scaled_states(scale):
    """A step is linear; where squares underflow the norm does, so only the smallest scales that keep it are taken."""
    m = 10
    dt = W.converging_dt(N, DR, L, m, ST, 0.06)
    x = W.smooth_state(N, DR, L, seed=4)
    if scale < 1e-150:                       # one row at the scale, the rest ordinary
        y = x.copy()
        y[L] *= scale
        assert rel_l2(_single(y, m, dt, "off"), _want(y, m, dt)) <= 1e-12
    else:
        assert rel_l2(_single(x * scale, m, dt, "off") / scale, _want(x, m, dt)) <= 1e-12


def test_underflowing_tail():
    """Amplitudes that fall through the subnormals keep their size pointwise."""
    n, l, m = 9001, 3, 8
    dt = W.converging_dt(n, 0.1, l, m, 5, 0.06)
    x = W.hydrogen_1s(n, 0.1, l)
    t = make(n, 0.1, l, 5, pulse=PULSE)
    t.set_state(x)
    t.time = 40.0
    t.propagate("lanczos", m, dt, 1)
    got = t.get_state()
    t.close()
    want = oracle.propagate(grid_of(n, 0.1, l, 5), x, "lanczos", m, dt, 1, t0=40.0, pulse=PULSE)[0]
    assert rel_l2(got, want) <= 1e-12
    r = W.radial_grid(n, 0.1)
    far = (r > 300) & (r < 700)
    assert np.all(np.abs(got[0, far] - want[0, far]) <= 1e-9 * np.abs(want[0, far]))

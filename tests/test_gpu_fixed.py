"""The fixed-point stencil of the FP64 length gauge (csrc/tdse_walk_fixed.cuh)
in the batch engine, at the sizes where its strips (60 columns, two a lane) and
chunks end, on random states (full grid-scale content in every partial wave),
against the oracle: 1e-12 relative L2 after one step at which the Krylov
propagator converges, the per-step bound of every FP64 path.  Also: values near
the limits of FP64, non-finite states, and grids whose coefficients the
fixed-point form cannot hold (the FP64 fallback)."""
import numpy as np
import pytest

import oracle
import tdse_workloads as W
from gpu_helpers import rel_l2

pytestmark = pytest.mark.gpu


def _spec(N, L, dr, m, st, E0=0.05):
    return dict(N=N, dr=dr, lmax=L, krylov=m, dt=W.converging_dt(N, dr, L, m, st, E0), E0=E0, omega=0.057, ncycles=2)


def _step(specs, states, st, t0=30.0):
    from paper_1308_1856_gb300 import Batch
    b = Batch(specs, stencil=st)
    for i, x in enumerate(states):
        b.set_state(i, x)
        b.set_time(i, t0)
    b.propagate(1)
    out = [b.get_state(i) for i in range(len(specs))]
    b.close()
    return out


def _want(s, x, st, t0=30.0):
    g = oracle.Grid(N=s["N"], h=s["dr"], L=s["lmax"], stencil=st)
    return oracle.propagate(g, x, "lanczos", s["krylov"], s["dt"], 1, t0=t0,
                            pulse=oracle.Pulse(E0=s["E0"], omega=s["omega"], ncycles=s["ncycles"]))[0]


@pytest.mark.parametrize("st", [3, 5])
def test_strip_and_chunk_edges(st):
    shapes = [(1, 0), (2, 1), (3, 0), (59, 3), (60, 4), (61, 5), (62, 33), (119, 2), (120, 31), (121, 40), (601, 7),
              (1203, 65)]
    specs = [_spec(N, L, 0.2 if i % 2 else 0.1, min(8, N * (L + 1)), st) for i, (N, L) in enumerate(shapes)]
    states = [W.random_state(N, L, seed=i) for i, (N, L) in enumerate(shapes)]
    for s, x, got in zip(specs, states, _step(specs, states, st)):
        want = _want(s, x, st)
        assert rel_l2(got, want) <= 1e-12, (s["N"], s["lmax"], rel_l2(got, want))


@pytest.mark.parametrize("scale", [1e-140, 1e140])
def test_scaled_states(scale):
    """H is linear: a state of another magnitude evolves to the scaled result."""
    s = _spec(500, 12, 0.1, 10, 5)
    x = W.smooth_state(500, 0.1, 12, seed=4)
    got = _step([s], [x * scale], 5)[0]
    assert rel_l2(got / scale, _want(s, x, 5)) <= 1e-12


def test_underflowing_tail():
    """The 1s state of a long box falls through the subnormals to zero; the tail
    stays finite and at its size, and the field's first step is the oracle's."""
    s = _spec(9001, 5, 0.1, 8, 5)
    x = W.hydrogen_1s(9001, 0.1, 5)
    assert np.any((np.abs(x[0]) > 0) & (np.abs(x[0]) < 1e-307)) and x[0, -1] == 0
    got, want = _step([s], [x], 5)[0], _want(s, x, 5)
    assert rel_l2(got, want) <= 1e-12
    r = W.radial_grid(9001, 0.1)
    far = (r > 300) & (r < 700)
    assert np.all(np.abs(got[0, far] - want[0, far]) <= 1e-9 * np.abs(want[0, far]))
    assert np.all(np.abs(got[0, r > 760]) < 1e-300)


def test_nonfinite_state_is_reported_and_stays_in_its_instance():
    from paper_1308_1856_gb300 import Batch, TDSEError
    s = _spec(300, 4, 0.1, 6, 5)
    good, bad = W.smooth_state(300, 0.1, 4, seed=1), W.smooth_state(300, 0.1, 4, seed=2)
    for v in (np.inf, np.nan):
        b = Batch([s, s], stencil=5)
        x = bad.copy()
        x[2, 140] = v
        b.set_state(0, good)
        b.set_state(1, x)
        b.propagate(1)
        ref = _step([s], [good], 5, t0=0.0)[0]
        assert np.array_equal(b.get_state(0), ref)
        assert not np.all(np.isfinite(b.get_state(1)))
        with pytest.raises(TDSEError):
            b.observables(1)
        b.close()


@pytest.mark.parametrize("dr,Z", [(9e-10, 1.0), (1e10, 1.0), (0.1, 1e14)])
def test_coefficients_outside_the_fixed_point_form(dr, Z):
    """Grid spacings and charges beyond the encoding run in FP64, as the oracle."""
    N, L, m = 130, 3, 4
    c0 = 30 / 24 / dr ** 2
    rho = 2.2 * c0 + L * (L + 1) / (2 * dr * dr) + Z / dr
    s = dict(N=N, dr=dr, lmax=L, krylov=m, dt=0.5 * m / rho, E0=0.0, omega=0.057, ncycles=2, Z=Z)
    x = W.random_state(N, L, seed=9)
    got = _step([s], [x], 5)[0]
    g = oracle.Grid(N=N, h=dr, L=L, stencil=5, Z=Z)
    want, _ = oracle.propagate(g, x, "lanczos", m, s["dt"], 1)
    assert rel_l2(got, want) <= 1e-12, rel_l2(got, want)

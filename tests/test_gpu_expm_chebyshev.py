"""The small exponential's Chebyshev series (csrc/tdse_small_expm.cuh) where it
begins and ends: half the spectrum's width times dt, z, from far below one to
both sides of the largest it takes, at every size of the matrix that matters,
shifted and scaled spectra, and one eigenvalue, against a 40-digit eigendecomposition.  Bound: test_gpu_expm.py's, 1e-13 + 4e-16 times the phases."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

pytest.importorskip("mpmath")


def _T(m, seed, shift=0.0, scale=1.0):
    rng = np.random.default_rng(seed)
    return scale * (rng.uniform(-1, 1, m) + shift), scale * rng.uniform(0.05, 1.0, m - 1)


def _dt(a, b, z):
    bb = np.concatenate([[0], b, [0]])
    rad = bb[:-1] + bb[1:]
    return z / (0.5 * ((a + rad).max() - (a - rad).min()))


@pytest.mark.parametrize("z", [1e-6, 0.1, 3.0, 12.0, 23.9, 24.1])
@pytest.mark.parametrize("m", [2, 12, 31, 32])
def test_series(m, z):
    from test_gpu_expm import _check
    a, b = _T(m, m)
    _check(a, b, _dt(a, b, z))


@pytest.mark.parametrize("shift,scale", [(0.0, 1e6), (50.0, 1.0), (-50.0, 1e-3), (3.0, 1e-12)])
def test_shifted_and_scaled_spectra(shift, scale):
    from test_gpu_expm import _check
    a, b = _T(10, 3, shift, scale)
    _check(a, b if scale > 1e-9 else 1e12 * b, _dt(a, b if scale > 1e-9 else 1e12 * b, 6.0))


@pytest.mark.parametrize("a", [0.0, 0.3, -1e5])
def test_one_value(a):
    from test_gpu_expm import _check
    _check(np.array([a]), np.array([]), 0.1)

"""The schedule's prefetch distance has no kernel: a captured step graph is
replayed whatever its value, and the autotuner leaves it as it is."""
import numpy as np
import pytest

import tdse_workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gauge", ["length", "velocity"])
def test_prefetch_rows_change_no_launch(gauge):
    from paper_1308_1856_gb300 import Batch, TDSEError
    N, L, m = 400, 5, 6
    s = dict(N=N, dr=0.1, lmax=L, krylov=m, dt=W.converging_dt(N, 0.1, L, m, 5, 0.05), E0=0.05, omega=0.057, ncycles=2,
             gauge=gauge)
    b = Batch([s, s], stencil=5)
    for i in range(2):
        b.set_state(i, W.smooth_state(N, 0.1, L, seed=i))
    for _ in range(4):
        b.propagate(1)
    steps = b.graph_steps
    now = b.schedule()
    for pf in (0, 3, 10):
        b.set_schedule(pf, now["stencil_blocks_per_sm"], now["elem_blocks_per_sm"], ring_rows=now["ring_rows"])
        b.propagate(1)
        steps += 1
        assert b.graph_steps == steps and b.schedule()["prefetch_rows"] == pf
    assert b.autotune()["prefetch_rows"] == 10
    with pytest.raises(TDSEError):
        b.set_schedule(4, 2, 2)
    assert np.all(np.isfinite(b.get_state(0)))
    b.close()

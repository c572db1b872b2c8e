"""tdse_batch_propagate_io plans its groups by the chunks one stencil launch takes at
once, which follow the schedule's blocks per SM: the same states, bitwise, for each."""
import numpy as np
import pytest

import tdse_workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("sblocks", [1, 2])
def test_groups_follow_the_schedule(precision, sblocks):
    import torch
    from paper_1308_1856_gb300 import Batch
    rng = np.random.default_rng(1)
    specs = []
    for _ in range(7):
        N, L, m = int(rng.integers(300, 4000)), int(rng.integers(2, 30)), int(rng.integers(4, 9))
        specs.append(dict(N=N, dr=0.1, lmax=L, krylov=m, dt=W.converging_dt(N, 0.1, L, m, 5, 0.05), E0=0.05, omega=0.057,
                          ncycles=2))
    states = [W.random_state(s["N"], s["lmax"], seed=i) for i, s in enumerate(specs)]
    flat = np.concatenate([x.ravel() for x in states])
    ref = Batch(specs, precision=precision)
    for i, x in enumerate(states):
        ref.set_state(i, x)
    ref.propagate(2)
    want = np.concatenate([ref.get_state(i).ravel() for i in range(len(specs))])
    ref.close()
    b = Batch(specs, precision=precision)
    b.set_schedule(6, sblocks, 2)
    src = torch.from_numpy(flat).pin_memory()
    out = torch.empty_like(src).pin_memory()
    for groups in (1, 3, 7):
        for i in range(len(specs)):
            b.set_time(i, 0.0)
        b.propagate_io(src.data_ptr(), out.data_ptr(), 2, groups)
        assert np.array_equal(out.numpy(), want), groups
    b.close()

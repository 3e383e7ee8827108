"""Step counts and checkpoint intervals of the adjoint near the range of their type."""
import numpy as np
import pytest

from paper_1202_6351_gb300 import lbm, workloads

pytestmark = pytest.mark.gpu

RATES = (1.1, 1.7, 1.7, 1.0, 1.2, 0.9)
MOST = 2 ** 63 - 1


def test_an_interval_beyond_the_run_is_one_segment():
    import torch

    nx, ny = 45, 38
    u, t = (torch.from_numpy(workloads.random_fields(s, nx, ny, u_amp=0.02)[1].copy()).cuda() for s in (5, 6))
    for store in (lbm.F64, lbm.F32):
        with lbm.Lattice(nx, ny, RATES, store=store) as L:
            want = L.adjoint_run(5, 5, u, t)
            for every in (6, MOST - 4, MOST):
                assert L.adjoint_workspace(5, every) == L.adjoint_workspace(5, 5)
                got = L.adjoint_run(5, every, u, t)
                assert got[0] == want[0]
                assert torch.equal(got[1], want[1]) and torch.equal(got[2], want[2])
                np.testing.assert_array_equal(got[3], want[3])


@pytest.mark.parametrize("nsteps,every", [(2 ** 62, 1), (MOST, 1), (MOST, MOST), (2 ** 57 - 1, 2 ** 57 - 1)])
def test_a_workspace_beyond_the_address_range_is_refused(nsteps, every):
    with lbm.Lattice(64, 64, RATES, store=lbm.F64) as L:
        with pytest.raises(lbm.LBMError) as e:
            L.adjoint_workspace(nsteps, every)
        assert e.value.code == lbm.LBM_ENOMEM

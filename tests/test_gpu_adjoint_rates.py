"""Rate gradients of the adjoint where the reverse step takes four rows per thread
(lattices of 2^20 nodes and more)."""
import numpy as np
import pytest

from paper_1202_6351_gb300 import lbm, workloads

pytestmark = pytest.mark.gpu

RATES = (1.1, 1.7, 1.7, 1.0, 1.2, 0.9)


def problem(nx, ny):
    import torch

    _, u = workloads.random_fields(5, nx, ny, u_amp=0.02)
    _, t = workloads.random_fields(6, nx, ny, u_amp=0.02)
    f = workloads.random_force_field(7, nx, ny, 1e-5)
    return [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (u, t, f)]


# The small lattice sums its nodes in other groups than the large one.  FP64: about 8 additions
# in a warp, 7 over time, 70 per thread and 7 per block of the last sum, each of relative error 1.1e-16
# of the sum of absolute values: 1e-14.  FP32: 8 additions in a warp at 6e-8, 5e-7.  The sum of
# absolute values is at most a few hundred times the largest of the six gradients.
@pytest.mark.parametrize("store,tol", [(lbm.F64, 1e-11), (lbm.F32, 1e-4)], ids=["f64", "f32"])
@pytest.mark.parametrize("tile,times", [((37, 41), (28, 26)), ((128, 64), (9, 15)), ((5, 3), (210, 351))],
                         ids=["1036x1066", "1152x960", "1050x1053"])
def test_rate_gradients_of_a_repeated_pattern_add_up(tile, times, store, tol):
    """A periodic lattice tiled with n copies of a small one has n times its rate gradients; the large
    ones have 2^20 nodes and more, with ragged last blocks in both directions, the small ones do not."""
    assert tile[0] * times[0] * tile[1] * times[1] >= 1 << 20
    fields = problem(*tile)
    out = []
    for k in ((1, 1), times):
        u, t, f = (a.tile((1, k[1], k[0])).contiguous() for a in fields)
        with lbm.Lattice(tile[0] * k[0], tile[1] * k[1], RATES, store=store) as L:
            L.set_force_field(f)
            out.append(L.adjoint_run(7, 3, u, t))
    n = times[0] * times[1]
    one, many = n * out[0][3], out[1][3]
    assert np.abs(one).max() > 0
    assert np.abs(many - one).max() <= tol * np.abs(one).max()

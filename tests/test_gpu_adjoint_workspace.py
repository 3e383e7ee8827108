"""lbm_adjoint_run_in: the adjoint in a workspace of the caller's, and the reverse
step's two block shapes (one node per thread, four rows per thread from 2^20 nodes
on) at sizes where their blocks are ragged."""
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


@pytest.mark.parametrize("store", [lbm.F64, lbm.F32], ids=["f64", "f32"])
@pytest.mark.parametrize("every", [1, 3, 20])
def test_workspace_of_the_callers_gives_the_same_gradients(store, every):
    import torch

    u, t, f = problem(45, 38)
    with lbm.Lattice(45, 38, RATES, store=store) as L:
        L.set_force_field(f)
        n = L.adjoint_workspace(10, every)
        ws = torch.full((n + 256,), 0xA5, dtype=torch.uint8, device="cuda")
        own = L.adjoint_run(10, every, u, t)
        given = L.adjoint_run(10, every, u, t, workspace=ws[:n])
        assert (ws[n:] == 0xA5).all()  # nothing beyond the size asked for
        assert own[0] == given[0]
        for a, b in zip(own[1:], given[1:]):
            np.testing.assert_array_equal(np.asarray(a.cpu() if hasattr(a, "cpu") else a),
                                          np.asarray(b.cpu() if hasattr(b, "cpu") else b))
        for bad in (ws[:n - 1], ws[1:n + 1]):  # too small; not 256-byte aligned
            with pytest.raises(lbm.LBMError) as e:
                L.adjoint_run(10, every, u, t, workspace=bad)
            assert e.value.code == lbm.LBM_EINVAL


@pytest.mark.parametrize("tile,times", [((37, 41), (28, 26)), ((5, 3), (7, 9)), ((1, 2), (33, 2)), ((130, 9), (1, 3))],
                         ids=lambda v: f"{v[0]}x{v[1]}")
def test_gradients_of_a_repeated_pattern_repeat(tile, times):
    """A periodic lattice tiled with copies of a smaller one computes the same values
    at every copy of a node, whatever block its thread sits in: start-field and force
    gradients repeat bit for bit, and the loss is that of one copy times their number
    up to the rounding of its FP64 sum.  37 x 28 by 41 x 26 nodes (over 2^20) takes four
    rows per thread, the rest one node per thread."""
    import torch

    fields = problem(*tile)
    out = []
    for k in ((1, 1), times):
        u, t, f = (a.tile((1, k[1], k[0])).contiguous() for a in fields)
        with lbm.Lattice(tile[0] * k[0], tile[1] * k[1], RATES, store=lbm.F32) as L:
            L.set_force_field(f)
            out.append(L.adjoint_run(7, 3, u, t))
    (loss0, gu0, gf0, _), (loss1, gu1, gf1, _) = out
    n = times[0] * times[1]
    assert torch.equal(gu0.tile((1, times[1], times[0])), gu1)
    assert torch.equal(gf0.tile((1, times[1], times[0])), gf1)
    assert abs(loss1 - n * loss0) <= 1e-12 * loss1

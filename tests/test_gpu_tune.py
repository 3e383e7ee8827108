"""lbm_tune on lattices that lbm_step steps on chip: the trials time the kernel that
calls of 8 or more steps run, and the lattice stays on it."""
import numpy as np
import pytest

from paper_1202_6351_gb300 import lbm, workloads

pytestmark = pytest.mark.gpu

OMEGAS = (1.1, 1.7, 1.7, 1.0, 1.2, 0.9)


@pytest.mark.parametrize("trial", [1, 20, 400])
@pytest.mark.parametrize("store", [lbm.F32, lbm.F16DEV, lbm.F64], ids=["f32", "f16", "f64"])
@pytest.mark.parametrize("shape", [(64, 64), (16, 16), (33, 47)], ids=["64x64", "16x16", "33x47"])
def test_tuning_keeps_a_small_lattice_on_chip(shape, store, trial):
    fits = -(-shape[1] // 16) * shape[0] <= (128 if store == lbm.F64 else 800)
    fields = workloads.random_fields(4, *shape, u_amp=0.03, rho_amp=0.01)
    with lbm.Lattice(*shape, OMEGAS, store=store) as L, lbm.Lattice(*shape, OMEGAS, store=store) as ref:
        L.init(*fields).step(3)
        ref.init(*fields).step(3)
        before = L.get_f()
        ms = L.tune(trial)
        np.testing.assert_array_equal(L.get_f(), before)
        assert L.time == 3
        admitted = {lbm.F64: (0,), lbm.F32: (0, 1, 3)}.get(store, (0, 1, 2, 3))
        assert all((ms[v] > 0) == (v in admitted) for v in range(lbm.NUM_VARIANTS))
        if fits:  # one kernel, one time for the variants that step on chip; variant 1 launches every step
            assert len({ms[v] for v in admitted if v != 1}) == 1
            assert L.info()["variant"] == 0 or trial == 1  # two trial steps of variant 1 are mostly launch
        ref.set_variant(L.info()["variant"])
        L.step(40)
        ref.step(40)
        np.testing.assert_array_equal(L.get_f(), ref.get_f())


@pytest.mark.parametrize("n", [150, 257, 400])
def test_f64_steps_have_one_block_shape(n):
    """The FP64 step ignores the block width: no trial of the others, and the default is kept."""
    with lbm.Lattice(n, n, OMEGAS, store=lbm.F64) as L:
        L.init(*workloads.random_fields(4, n, n, u_amp=0.03, rho_amp=0.01))
        width = L.info()["block_x"]
        assert L.tune(20)[0] > 0
        assert L.info()["block_x"] == width

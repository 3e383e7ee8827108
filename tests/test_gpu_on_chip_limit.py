"""Which lattices lbm_step advances on chip: the tuner reports one time for variants 0 and 3 where they
are one kernel, and a time for each where every step is launched."""
import pytest

from paper_1202_6351_gb300 import lbm, workloads

pytestmark = pytest.mark.gpu

OMEGAS = (1.1, 1.7, 1.7, 1.0, 1.2, 0.9)


@pytest.mark.parametrize("shape,store,force,stochastic,chip", [
    ((800, 16), lbm.F32, False, False, True), ((801, 16), lbm.F32, False, False, False),
    ((720, 16), lbm.F32, True, False, True), ((721, 16), lbm.F32, True, False, False),
    ((720, 16), lbm.F32, False, True, True), ((721, 16), lbm.F32, False, True, False),
    ((512, 16), lbm.F32, True, True, True), ((513, 16), lbm.F32, True, True, False),
    ((720, 16), lbm.F16DEV, True, True, True), ((721, 16), lbm.F16DEV, True, True, False),
    ((112, 112), lbm.F32, True, True, False), ((64, 64), lbm.F32, True, True, True),
])
def test_long_updates_step_on_chip_only_where_that_is_faster(shape, store, force, stochastic, chip):
    with lbm.Lattice(*shape, OMEGAS, store=store) as L:
        if force:
            L.set_force_field(workloads.random_force_field(3, *shape, 1e-6))
        if stochastic:
            L.set_rounding(lbm.ROUND_STOCHASTIC, 5)
        ms = L.init().tune(50)
        assert ms[0] > 0 and ms[3] > 0
        assert (ms[0] == ms[3]) == chip

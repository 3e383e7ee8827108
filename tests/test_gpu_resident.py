"""Small lattices stepped on chip (csrc/lbm_resident.cuh: 8 or more steps of one
call in one launch) against one launch per step: the states are bit for bit the
same, for every collision, edge, force, storage and rounding, from even and odd
steps, at the sizes where slabs of rows are uneven, a cluster has fewer CTAs than
16, and the lattice just fits (800 nodes per CTA) or just does not."""
import numpy as np
import pytest

from paper_1202_6351_gb300 import lbm, workloads

pytestmark = pytest.mark.gpu

P, BB, MW = lbm.PERIODIC, lbm.BOUNCEBACK, lbm.MOVING_WALL
EDGES = {
    "periodic": ((P, P, P, P), (0, 0, 0, 0)),
    "cavity": ((MW, BB, MW, MW), (0.02, 0, -0.03, 0.1)),
    "channel": ((P, P, BB, MW), (0, 0, 0, 0.05)),
}
SHAPES = [(1, 1), (5, 1), (1, 40), (2, 2), (4, 4), (37, 5), (33, 15), (16, 16), (31, 17), (26, 26), (101, 101), (112, 112),
          (800, 16), (801, 16), (50, 256), (50, 257), (3, 4000)]


@pytest.fixture(scope="module", autouse=True)
def cuda():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    torch.cuda.set_device(0)
    yield


def run(shape, edges, model, store, force, stochastic, calls):
    nx, ny = shape
    kinds, speeds = EDGES[edges]
    rho, u = workloads.random_fields(nx + 7 * ny, nx, ny, u_amp=0.03, rho_amp=0.01)
    uniform = (2e-5, -1e-5) if force == "uniform" else (0.0, 0.0)
    with lbm.Lattice(nx, ny, (1.1, 1.7, 1.7, 1.0, 1.2, 0.9), force=uniform, edges=kinds, wall_u=speeds, model=model,
                     store=store) as L:
        if force == "field":
            L.set_force_field(workloads.random_force_field(3, nx, ny, 1e-5))
        if stochastic:
            L.set_rounding(lbm.ROUND_STOCHASTIC, 11)
        L.init(rho, u)
        out = []
        for n in calls:
            L.step(n)
            out.append(L.get_f())
        return out


@pytest.mark.parametrize("stochastic", [False, True], ids=["nearest", "stochastic"])
@pytest.mark.parametrize("store", [lbm.F32, lbm.F16DEV, lbm.BF16DEV], ids=["f32", "f16", "bf16"])
@pytest.mark.parametrize("edges", list(EDGES))
@pytest.mark.parametrize("shape", SHAPES, ids=[f"{a}x{b}" for a, b in SHAPES])
def test_on_chip_steps_are_bitwise_equal_to_single_launches(shape, edges, store, stochastic):
    k = SHAPES.index(shape) + list(EDGES).index(edges) + int(store)
    model = (lbm.CASCADED, lbm.BGK, lbm.RAWMRT)[k % 3]
    force = ("none", "uniform", "field")[(k // 2) % 3]
    # 9 and 16 steps in one call each (the second from an odd step), against calls of one step
    whole = run(shape, edges, model, store, force, stochastic, (9, 16))
    single = run(shape, edges, model, store, force, stochastic, (1,) * 25)
    for a, b in zip(whole, (single[8], single[24])):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("model", [lbm.CASCADED, lbm.BGK, lbm.RAWMRT], ids=["cascaded", "bgk", "rawmrt"])
@pytest.mark.parametrize("force", ["none", "uniform", "field"])
def test_on_chip_steps_of_every_collision_and_force(model, force):
    for edges in EDGES:
        whole = run((45, 30), edges, model, lbm.F32, force, False, (40,))
        single = run((45, 30), edges, model, lbm.F32, force, False, (1,) * 40)
        np.testing.assert_array_equal(whole[0], single[-1])


def test_divergence_checks_fall_on_the_same_steps():
    """The check runs at every multiple of `every` steps also when the steps between
    two checks are one launch."""
    sums = []
    for calls in ((50,), (1,) * 50):
        with lbm.Lattice(40, 30, (1.0, 1.9, 1.9, 1.0, 1.0, 1.0), edges=EDGES["cavity"][0], wall_u=EDGES["cavity"][1]) as L:
            L.init()
            L.set_check(20, 1e-3)
            for n in calls:
                L.step(n)
            sums.append((L.time, L.stats().tolist()))
    assert sums[0] == sums[1]
    for n in (200, 1):  # a start far outside the model's range: reported at the first check
        with lbm.Lattice(40, 30, (1.0, 1.99, 1.99, 1.0, 1.0, 1.0), model=lbm.BGK) as L:
            L.init(*workloads.random_fields(1, 40, 30, u_amp=0.6, rho_amp=0.0))
            L.set_check(20, 1e-9)
            with pytest.raises(lbm.LBMError) as err:
                for _ in range(200 // n):
                    L.step(n)
            assert err.value.code == lbm.LBM_EDIVERGED
            assert L.time % 20 == 0


# FP64: 128 nodes per CTA
F64_SHAPES = [(1, 1), (5, 1), (128, 1), (129, 1), (1, 40), (2, 2), (4, 4), (4, 32), (37, 5), (33, 15), (31, 17), (16, 128), (64, 32),
              (42, 48), (128, 16), (129, 16), (3, 600)]


@pytest.mark.parametrize("force", ["none", "uniform", "field"])
@pytest.mark.parametrize("model", [lbm.CASCADED, lbm.BGK, lbm.RAWMRT], ids=["cascaded", "bgk", "rawmrt"])
@pytest.mark.parametrize("shape", F64_SHAPES, ids=[f"{a}x{b}" for a, b in F64_SHAPES])
def test_on_chip_f64_steps_are_bitwise_equal_to_single_launches(shape, model, force):
    for edges in EDGES:
        whole = run(shape, edges, model, lbm.F64, force, False, (9, 16))
        single = run(shape, edges, model, lbm.F64, force, False, (1,) * 25)
        for a, b in zip(whole, (single[8], single[24])):
            np.testing.assert_array_equal(a, b)

"""Variant 3 with up to four steps per launch (csrc/lbm_multi.cuh, unforced
cascaded collision, round to nearest) against one step per launch: the states
are bit for bit the same.  Sizes sit at the edges of the 32 x 16 and 56 x 40
tiles and of the size rule between them, and below the four-node halo; step
counts cover launches of four and two steps and single steps at either end."""
import numpy as np
import pytest

from paper_1202_6351_gb300 import lbm, workloads

pytestmark = pytest.mark.gpu

P, BB, MW = lbm.PERIODIC, lbm.BOUNCEBACK, lbm.MOVING_WALL
EDGES = {
    "periodic": ((P, P, P, P), (0, 0, 0, 0)),
    "cavity": ((MW, BB, MW, MW), (0.02, 0, -0.03, 0.1)),
    "channel_x": ((P, P, BB, MW), (0, 0, 0, 0.05)),
    "channel_y": ((BB, MW, P, P), (0, 0.04, 0, 0)),
}
SHAPES = [(4, 4), (5, 7), (31, 17), (32, 16), (33, 18), (65, 5), (600, 599),            # 32 x 16 tiles
          (600, 600), (617, 603), (672, 560), (673, 561), (7, 52001), (9002, 41)]       # 56 x 40 tiles


@pytest.fixture(scope="module", autouse=True)
def cuda():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    torch.cuda.set_device(0)
    yield


@pytest.mark.parametrize("store", [lbm.F32, lbm.F16DEV, lbm.BF16DEV], ids=["f32", "f16", "bf16"])
@pytest.mark.parametrize("edges", list(EDGES))
@pytest.mark.parametrize("shape", SHAPES, ids=[f"{a}x{b}" for a, b in SHAPES])
def test_multi_step_launches_are_bitwise_equal_to_single_steps(shape, edges, store):
    nx, ny = shape
    kinds, speeds = EDGES[edges]
    rho, u = workloads.random_fields(nx + 7 * ny, nx, ny, u_amp=0.03, rho_amp=0.01)
    states = {}
    for variant in (0, 3):
        with lbm.Lattice(nx, ny, (1.1, 1.7, 1.7, 1.0, 1.2, 0.9), edges=kinds, wall_u=speeds, store=store) as L:
            L.set_variant(variant).init(rho, u)
            states[variant] = []
            for n in (4, 2, 1, 7, 10):  # launches of 4; 2; 1; 1 + 4 + 2; 4 + 4 + 2 steps
                L.step(n)
                states[variant].append(L.get_f())
            assert L.time == 24
    for a, b in zip(states[0], states[3]):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("start", [0, 1], ids=["even_start", "odd_start"])
def test_batches_of_unforced_lattices_take_four_steps_per_launch(start):
    """A batch whose lattices all take the multi-step tile, against the lattices
    stepped alone; a force set on one lattice between calls moves the batch to the
    two-step tiles and its removal back."""
    om = (1.1, 1.7, 1.7, 1.0, 1.2, 0.9)
    specs = [(64, 64, lbm.F32, "periodic"), (57, 41, lbm.F16DEV, "cavity"), (113, 37, lbm.F32, "channel_x"),
             (4, 5, lbm.BF16DEV, "periodic"), (300, 7, lbm.F16DEV, "channel_y"), (56, 80, lbm.F32, "cavity")]

    def make(i):
        nx, ny, store, edges = specs[i]
        L = lbm.Lattice(nx, ny, om, edges=EDGES[edges][0], wall_u=EDGES[edges][1], store=store)
        return L.init(*workloads.random_fields(i, nx, ny, u_amp=0.03, rho_amp=0.01)).step(start)

    alone, batched = ([make(i) for i in range(len(specs))] for _ in range(2))
    with lbm.Batch(batched) as B:
        B.set_graph_steps(20)  # two launches of four steps, twice per replay
        B.set_two_step(True)
        for force, tile in (((0.0, 0.0), (56, 40)), ((1e-5, 0.0), (64, 16)), ((0.0, 0.0), (56, 40))):
            for L in (alone[0], batched[0]):
                L.set_force(force)
            for n in (29, 6, 2):
                B.step(n)
                for L in alone:
                    L.step(n)
            assert B.info()["tile"] == tile
            B.sync()
            for i, (a, b) in enumerate(zip(alone, batched)):
                assert a.time == b.time
                np.testing.assert_array_equal(a.get_f(), b.get_f(), err_msg=f"lattice {i}")
    for L in alone + batched:
        L.close()

"""Variant 3 with several steps per launch at the lines between its tile shapes (csrc/lbm_multi.cuh:
32 x 16 tiles, 56 x 40 tiles, and those with 384 threads for 16-bit storage): bit for bit single steps."""
import numpy as np
import pytest

from paper_1202_6351_gb300 import lbm, workloads

pytestmark = pytest.mark.gpu

P, BB, MW = lbm.PERIODIC, lbm.BOUNCEBACK, lbm.MOVING_WALL
EDGES = {"periodic": ((P, P, P, P), (0, 0, 0, 0)), "cavity": ((MW, BB, MW, MW), (0.02, 0, -0.03, 0.1)),
         "channel": ((P, P, BB, MW), (0, 0, 0, 0.05))}
# 450 and 465 small tiles; 130 and 153 large ones of 152; 304 and 306; ragged, narrow and flat lattices
SHAPES = [(480, 480), (496, 480), (520, 520), (17 * 56, 9 * 40), (19 * 56, 16 * 40), (18 * 56, 17 * 40), (57, 2000), (9002, 44),
          (20, 9000), (1000, 401)]


@pytest.mark.parametrize("store", [lbm.F32, lbm.F16DEV, lbm.BF16DEV], ids=["f32", "f16", "bf16"])
@pytest.mark.parametrize("edges", list(EDGES))
@pytest.mark.parametrize("shape", SHAPES, ids=[f"{a}x{b}" for a, b in SHAPES])
def test_tile_shapes_are_bitwise_equal_to_single_steps(shape, edges, store):
    nx, ny = shape
    kinds, speeds = EDGES[edges]
    rho, u = workloads.random_fields(nx + 3 * ny, nx, ny, u_amp=0.03, rho_amp=0.01)
    states = []
    for variant in (0, 3):
        with lbm.Lattice(nx, ny, (1.1, 1.7, 1.7, 1.0, 1.2, 0.9), edges=kinds, wall_u=speeds, store=store) as L:
            L.set_variant(variant).init(rho, u)
            states.append([])
            for n in (6, 9):
                L.step(n)
                states[-1].append(L.get_f())
    for a, b in zip(*states):
        np.testing.assert_array_equal(a, b)

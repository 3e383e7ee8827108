"""The tiles a batch takes several steps on: four steps on 56 x 40 tiles where they cost less than two on
64 x 16, by the sizes and edges of its lattices; the states are those of the lattices stepped alone."""
import numpy as np
import pytest

from paper_1202_6351_gb300 import lbm, workloads

pytestmark = pytest.mark.gpu

P, BB, MW = lbm.PERIODIC, lbm.BOUNCEBACK, lbm.MOVING_WALL
EDGES = {"periodic": ((P, P, P, P), (0, 0, 0, 0)), "cavity": ((MW, BB, MW, MW), (0.02, 0, -0.03, 0.1))}
OMEGAS = (1.1, 1.7, 1.7, 1.0, 1.2, 0.9)


@pytest.mark.parametrize("store", [lbm.F32, lbm.F16DEV], ids=["f32", "f16"])
@pytest.mark.parametrize("count,shapes,edges,tile", [
    (60, [(64, 64)], "periodic", (64, 16)), (60, [(57, 57)], "periodic", (64, 16)), (60, [(64, 64)], "cavity", (56, 40)),
    (4, [(64, 64)], "periodic", (56, 40)), (80, [(48, 48)], "periodic", (56, 40)), (60, [(72, 72)], "periodic", (56, 40)),
    (40, [(130, 130), (64, 64), (33, 90)], "periodic", (56, 40)), (200, [(16, 16), (57, 41)], "cavity", (56, 40)),
])
def test_tiles_of_a_batch_and_its_states(count, shapes, edges, tile, store):
    def make(i):
        nx, ny = shapes[i % len(shapes)]
        L = lbm.Lattice(nx, ny, OMEGAS, edges=EDGES[edges][0], wall_u=EDGES[edges][1], store=store)
        return L.init(*workloads.random_fields(i, nx, ny, u_amp=0.03, rho_amp=0.01))

    alone, batched = ([make(i) for i in range(count)] for _ in range(2))
    with lbm.Batch(batched) as B:
        B.set_two_step(True)
        B.set_graph_steps(16)
        B.step(41)
        B.sync()
        assert B.info()["tile"] == tile
        for i, (a, b) in enumerate(zip(alone, batched)):
            np.testing.assert_array_equal(a.step(41).get_f(), b.get_f(), err_msg=f"lattice {i}")
    for L in alone + batched:
        L.close()

"""Two host threads, each stepping a lattice of its own: the lattices differ in size
and use the same kernels, and neither may disturb the other's launches."""
import threading

import numpy as np
import pytest

from paper_1202_6351_gb300 import lbm, workloads

pytestmark = pytest.mark.gpu

OMEGAS = (1.1, 1.7, 1.7, 1.0, 1.2, 0.9)


@pytest.mark.parametrize("store,shapes", [(lbm.F32, ((16, 16), (112, 112))), (lbm.F16DEV, ((5, 40), (800, 16))),
                                          (lbm.F64, ((8, 8), (42, 48)))], ids=["f32", "f16", "f64"])
def test_small_lattices_of_two_threads(store, shapes):
    """Calls of 8 steps take the on-chip kernel, whose shared memory depends on the lattice."""
    import torch

    calls, errors, states = 2000, [], {}

    def work(shape):
        try:
            torch.cuda.set_device(0)
            stream = torch.cuda.Stream()
            with lbm.Lattice(*shape, OMEGAS, store=store, stream=stream.cuda_stream) as L:
                L.init(*workloads.random_fields(3, *shape, u_amp=0.03, rho_amp=0.01))
                for _ in range(calls):
                    L.step(8)
                states[shape] = L.get_f()
        except Exception as e:  # reported by the main thread
            errors.append(f"{shape}: {e}")

    threads = [threading.Thread(target=work, args=(s,)) for s in shapes]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for shape in shapes:  # and the same states as alone
        with lbm.Lattice(*shape, OMEGAS, store=store) as L:
            L.init(*workloads.random_fields(3, *shape, u_amp=0.03, rho_amp=0.01)).step(8 * calls)
            np.testing.assert_array_equal(L.get_f(), states[shape])

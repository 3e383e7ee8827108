"""CUDA-graph replay in lbm_step on lattices too large for the on-chip kernel
(ceil(ny / 16) * nx > 800, so 8 or more steps of a call do reach the graph): the
states do not depend on it, and switching the divergence check between calls,
which changes what a replay holds under variant 3, keeps states and step count."""
import numpy as np
import pytest

from paper_1202_6351_gb300 import lbm, workloads

pytestmark = pytest.mark.gpu

P, BB, MW = lbm.PERIODIC, lbm.BOUNCEBACK, lbm.MOVING_WALL
OMEGAS = (1.1, 1.7, 1.7, 1.0, 1.2, 0.9)
EDGES = {"periodic": ((P, P, P, P), (0, 0, 0, 0)), "cavity": ((MW, BB, MW, MW), (0.02, 0, -0.03, 0.1))}


@pytest.fixture(scope="module", autouse=True)
def cuda():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    torch.cuda.set_device(0)
    yield


def lattice(nx, ny, store, model=lbm.CASCADED, edges="periodic", force=(0.0, 0.0), stochastic=False):
    assert -(-ny // 16) * nx > 800  # steps launch by launch
    kinds, speeds = EDGES[edges]
    L = lbm.Lattice(nx, ny, OMEGAS, force=force, edges=kinds, wall_u=speeds, model=model, store=store)
    if stochastic:
        L.set_rounding(lbm.ROUND_STOCHASTIC, 5)
    return L.init(*workloads.random_fields(nx + 7 * ny, nx, ny, u_amp=0.03, rho_amp=0.01))


KINDS = {  # lattices whose variant 3 replays two-step launches
    "rawmrt": dict(store=lbm.F32, model=lbm.RAWMRT),
    "bgk_f16": dict(store=lbm.F16DEV, model=lbm.BGK),
    "forced": dict(store=lbm.F32, force=(2e-5, -1e-5)),
    "stochastic": dict(store=lbm.F32, stochastic=True),
    "stochastic_bf16": dict(store=lbm.BF16DEV, stochastic=True, edges="cavity"),
}


@pytest.mark.parametrize("checks", [(0, 100, 0), (100, 0, 100)], ids=["on_between", "off_between"])
@pytest.mark.parametrize("graph_steps", [6, 50])
@pytest.mark.parametrize("kind", list(KINDS))
def test_switching_the_check_recaptures_the_step_graph(kind, graph_steps, checks):
    """graph_steps = 2 mod 4: a replay of variant 3 holds graph_steps - 2 steps with
    the check off and graph_steps with it on."""
    def run(variant, graph, calls):
        with lattice(257, 129, **KINDS[kind]) as L:
            L.set_variant(variant).set_graph_steps(graph)
            out = []
            for every in checks:
                L.set_check(every, 1e-3)
                for n in calls:
                    L.step(n)
                out.append((L.time, L.get_f()))
            return out

    whole = run(3, graph_steps, (100,))
    single = run(0, 0, (1,) * 100)
    for (ta, fa), (tb, fb) in zip(whole, single):
        assert ta == tb
        np.testing.assert_array_equal(fa, fb)


@pytest.mark.parametrize("edges,force", [("periodic", (0.0, 0.0)), ("cavity", (0.0, 0.0)), ("cavity", (2e-5, 1e-5))])
@pytest.mark.parametrize("stochastic", [False, True], ids=["nearest", "stochastic"])
@pytest.mark.parametrize("store", [lbm.F32, lbm.F16DEV, lbm.BF16DEV, lbm.F64], ids=["f32", "f16", "bf16", "f64"])
@pytest.mark.parametrize("shape", [(257, 70), (403, 45)], ids=["257x70", "403x45"])
def test_replays_are_bitwise_equal_to_single_launches(shape, store, stochastic, edges, force):
    """Every variant that rounds alike, at two replay lengths, from odd and even steps and
    across a change of rates."""
    if stochastic and store == lbm.F64:
        pytest.skip("FP64 storage rounds to nearest only")

    def run(variant, graph, split):
        with lattice(*shape, store, edges=edges, force=force, stochastic=stochastic) as L:
            L.set_variant(variant).set_graph_steps(graph)
            out = []
            for n in (3, 37, 66):
                for k in ([1] * n if split else [n]):
                    L.step(k)
                out.append(L.get_f())
                L.set_omegas((1.0, 1.5, 1.5, 1.0, 1.1, 1.0))
            assert L.time == 106
            return out

    ref = run(0, 0, True)
    variants = {lbm.F64: (0,), lbm.F32: (0, 3)}.get(store, (0, 2, 3))
    for variant in variants:
        for graph in (8, 64):
            for k, (a, b) in enumerate(zip(run(variant, graph, False), ref)):
                np.testing.assert_array_equal(a, b, err_msg=f"variant {variant}, graph {graph}, chunk {k}")

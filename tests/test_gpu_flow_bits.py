"""Flow steps give the same bits however they are launched: several to a launch, one
at a time, inside a replayed graph or outside, on grids of one region, several, and
strips that go node by node.  The collision is one sequence of operations, rounded
alike, and wall nodes take the values of the wall pass."""
import numpy as np
import pytest

from paper_2209_01444_gb300 import workloads as W

pytestmark = pytest.mark.gpu

WALLS = {
    "periodic": ("periodic",) * 4,
    "channel": ("inflow", "outflow", "symmetry", "symmetry"),
    "noslip": ("periodic", "periodic", "noslip", "noslip"),
    "tube": ("symmetry", "noslip", "periodic", "periodic"),
}


def _run(nx, ny, walls, storage, n_sub, calls, flow):
    from paper_2209_01444_gb300 import lbm as L

    p = W.thermosolutal_params(nx, ny, bc=WALLS[walls], u_in=(0.1, 0.02), gbetaT=W.GBETA_T, gbetaC=W.GBETA_C,
                               force=(2e-4, 1e-4), n_sub=n_sub)
    sim = L.Simulation(p, storage=storage)
    sim.init_seeds(np.array([[0.5 * nx, 0.5 * ny, min(6.0, 0.3 * min(nx, ny)), 0.1]]), -0.2, -0.55)
    for n in calls:
        (sim.step_flow if flow else sim.step)(n)
    return sim.state()


@pytest.mark.parametrize("nx,ny", [(5, 33), (57, 25), (131, 70), (20000, 4)])
@pytest.mark.parametrize("walls", sorted(WALLS))
@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
def test_flow_steps(nx, ny, walls, storage):
    want = _run(nx, ny, walls, storage, 1, (1,) * 9, True)
    for calls in ((9,), (2, 7), (4, 5)):
        assert np.array_equal(_run(nx, ny, walls, storage, 1, calls, True), want), calls


# 32 steps are two replayed graphs, whose flow steps may go node by node where those
# of direct launches go several at a time
@pytest.mark.parametrize("n_sub", [3, 6])
@pytest.mark.parametrize("walls", sorted(WALLS))
def test_coupled_steps(walls, n_sub):
    want = _run(60, 41, walls, "fp32", n_sub, (1,) * 35, False)
    for calls in ((35,), (20, 15)):
        assert np.array_equal(_run(60, 41, walls, "fp32", n_sub, calls, False), want), calls

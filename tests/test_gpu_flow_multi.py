"""Flow steps taken several to a launch against the same steps one at a time.

``step_flow(n)`` keeps regions of the grid on chip for several steps; n calls
of ``step_flow(1)`` go node by node with the wall pass after each.  Both run
the same operations, so they differ by rounding alone: in FP32 by a few units
in the last place per step (2^-23 of populations of order one against speeds of
order 0.1: 1e-5 of the largest speed over ten steps), in 16-bit storage by
single roundings that fall the other way (2^-11 and 2^-8 of a deviation).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TOL = {"fp32": 1e-5, "fp16": 2e-3, "bf16": 3e-2}
WALLS = {
    "periodic": ("periodic",) * 4,
    "channel": ("inflow", "outflow", "symmetry", "symmetry"),
    "noslip": ("periodic", "periodic", "noslip", "noslip"),
    "tube": ("symmetry", "noslip", "periodic", "periodic"),
}


def _sim(L, W, nx, ny, walls, storage):
    p = W.thermosolutal_params(nx, ny, bc=WALLS[walls], u_in=(0.5, 0.1), gbetaT=W.GBETA_T, gbetaC=W.GBETA_C,
                               force=(2e-4, 1e-4))
    sim = L.Simulation(p, storage=storage)
    fields, _ = W.random_fields(nx, ny, 11, u_amp=0.5)
    sim.init_fields(fields)
    return sim


# regions are 64 x 32 nodes with rings of 2, 4 or 5: grids below one region, at
# its written size and one node more, and several regions with ragged ends
@pytest.mark.parametrize("nx,ny", [(4, 4), (5, 33), (56, 24), (57, 25), (60, 28), (109, 45), (131, 70)])
@pytest.mark.parametrize("walls", sorted(WALLS))
def test_steps_together_equal_steps_alone(gpu_lib, nx, ny, walls):
    L, W = gpu_lib
    for n in (2, 4, 5, 9):
        a, b = _sim(L, W, nx, ny, walls, "fp32"), _sim(L, W, nx, ny, walls, "fp32")
        a.step_flow(n)
        for _ in range(n):
            b.step_flow(1)
        fa, fb = a.fields(("ux", "uy", "p")), b.fields(("ux", "uy", "p"))
        speed = np.hypot(fb["ux"], fb["uy"]).max()
        for name in ("ux", "uy"):
            assert np.abs(fa[name] - fb[name]).max() <= TOL["fp32"] * speed, (name, n)
        assert np.abs(fa["p"] - fb["p"]).max() <= TOL["fp32"] * max(np.abs(fb["p"]).max(), speed), n


@pytest.mark.parametrize("storage", ["fp16", "bf16"])
@pytest.mark.parametrize("walls", ["channel", "noslip"])
def test_16_bit_storage(gpu_lib, storage, walls):
    L, W = gpu_lib
    a, b = _sim(L, W, 131, 70, walls, storage), _sim(L, W, 131, 70, walls, storage)
    a.step_flow(9)
    for _ in range(9):
        b.step_flow(1)
    fa, fb = a.fields(("ux", "uy")), b.fields(("ux", "uy"))
    speed = np.hypot(fb["ux"], fb["uy"]).max()
    for name in ("ux", "uy"):
        assert np.abs(fa[name] - fb[name]).max() <= TOL[storage] * speed, name


# away from walls 16-bit storage steps to the bit as one step at a time does: the
# collision is the single step's, whatever the steps of a launch (2, 4 and 5)
@pytest.mark.parametrize("storage", ["fp16", "bf16"])
@pytest.mark.parametrize("n", [2, 8, 15])
def test_16_bit_steps_are_the_single_steps_bits(gpu_lib, storage, n):
    L, W = gpu_lib
    a, b = _sim(L, W, 109, 45, "periodic", storage), _sim(L, W, 109, 45, "periodic", storage)
    a.step_flow(n)
    for _ in range(n):
        b.step_flow(1)
    fa, fb = a.fields(("ux", "uy", "p")), b.fields(("ux", "uy", "p"))
    for name in fa:
        assert np.array_equal(fa[name], fb[name]), name


@pytest.fixture(scope="module")
def gpu_lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2209_01444_gb300 import lbm as L
    from paper_2209_01444_gb300 import workloads as W

    L.load()
    return L, W

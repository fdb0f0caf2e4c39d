"""Flow steps next to walls: four to a launch, launches after the first
(which update the walls that the launch before left out) and launches of fewer
steps than the region's rings allow among them, against the same steps one at a
time.  On grids of one wave 3, 7 and 8 steps are launches of 3, 4 + 3 and 4 + 4; at
1024^2, several waves, 14 steps are launches of 4, 4, 3 and 3.  And steps of long strips,
which go node by node.

FP32 differs by rounding: a few units (2^-23 of populations of order one, against
speeds of order 0.1: 1.2e-6 each) per step, two of them allowed.  16-bit storage:
single roundings of a deviation, 2e-3 (FP16) and 3e-2 (BF16) of the largest speed.
A wall or rim node taken from the wrong place is off by O(0.1)."""
import numpy as np
import pytest

from paper_2209_01444_gb300 import workloads as W

pytestmark = pytest.mark.gpu

WALLS = {
    "channel": ("inflow", "outflow", "symmetry", "symmetry"),
    "noslip": ("periodic", "periodic", "noslip", "noslip"),
    "tube": ("symmetry", "noslip", "periodic", "periodic"),
}


def _compare(nx, ny, walls, storage, n, tol):
    from paper_2209_01444_gb300 import lbm as L

    p = W.thermosolutal_params(nx, ny, bc=WALLS[walls], u_in=(0.5, 0.1), gbetaT=W.GBETA_T, gbetaC=W.GBETA_C,
                               force=(2e-4, 1e-4))
    fields, _ = W.random_fields(nx, ny, 11, u_amp=0.5)
    out = []
    for calls in ((n,), (1,) * n):
        sim = L.Simulation(p, storage=storage)
        sim.init_fields(fields)
        for k in calls:
            sim.step_flow(k)
        out.append(sim.fields(("ux", "uy", "p")))
    a, b = out
    speed = np.hypot(b["ux"], b["uy"]).max()
    for name in ("ux", "uy"):
        assert np.abs(a[name] - b[name]).max() <= tol * speed, name
    if storage == "fp32":
        assert np.abs(a["p"] - b["p"]).max() <= tol * max(np.abs(b["p"]).max(), speed)


# regions are 64 x 32 nodes of which 56 x 24 are written
@pytest.mark.parametrize("nx,ny", [(5, 33), (56, 24), (57, 25), (60, 28), (109, 45), (131, 70)])
@pytest.mark.parametrize("walls", sorted(WALLS))
@pytest.mark.parametrize("n", [3, 7, 8])
def test_four_steps_a_launch(nx, ny, walls, n):
    _compare(nx, ny, walls, "fp32", n, 2.4e-6 * n)


@pytest.mark.parametrize("walls", sorted(WALLS))
@pytest.mark.parametrize("storage,tol", [("fp16", 2e-3), ("bf16", 3e-2)])
@pytest.mark.parametrize("n", [3, 7, 8])
def test_four_steps_a_launch_16_bit(walls, storage, tol, n):
    _compare(131, 70, walls, storage, n, tol)


def test_several_waves():
    _compare(1024, 1024, "channel", "fp32", 14, 2.4e-6 * 14)


# strips of which a region covers a small part go node by node, each step but the
# first updating the walls that the step before left out; corners among them
@pytest.mark.parametrize("nx,ny,walls", [(20000, 4, "channel"), (20001, 5, "noslip"), (20000, 6, "tube"),
                                         (4, 9000, "noslip")])
@pytest.mark.parametrize("storage,tol", [("fp32", 2.4e-6 * 3), ("fp16", 2e-3), ("bf16", 3e-2)])
def test_long_strips(nx, ny, walls, storage, tol):
    _compare(nx, ny, walls, storage, 3, tol)

"""Steps of one call update wall rows and columns as they load them (grids of
up to 2^20 nodes; larger ones the columns alone); profiled steps run the wall
passes after every step.  Both states agree to rounding of the same operations
in another kernel: 1e-5 with FP32 storage, single storage roundings (a deviation
near 1 in FP16 at a scale of 16: 1e-3) otherwise.  A wall cell taken from the
wrong node is off by O(0.1)."""
import numpy as np
import pytest

from paper_2209_01444_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL = {"fp32": 1e-5, "fp16": 4e-3}
WALLS = {"open": ("inflow", "outflow", "symmetry", "symmetry"), "rows": ("periodic", "periodic", "noslip", "dirichlet"),
         "box": ("noslip", "dirichlet", "symmetry", "noslip")}


# tiles are 32 x 4: both row walls in one tile (ny = 4), a wall row alone in the
# last tile (ny = 5, 9), in the halo of the last but one, ragged columns
@pytest.mark.parametrize("nx,ny", [(4, 4), (33, 5), (34, 9), (64, 6), (31, 7)])
@pytest.mark.parametrize("walls", sorted(WALLS))
@pytest.mark.parametrize("storage", ["fp32", "fp16"])
def test_small_grids(nx, ny, walls, storage):
    _check(nx, ny, walls, storage, (3, 18))


def test_columns_alone_on_a_large_grid():
    _check(1040, 1032, "open", "fp32", (3,))


def _check(nx, ny, walls, storage, counts):
    from paper_2209_01444_gb300 import lbm as L

    p = W.thermosolutal_params(nx, ny, bc=WALLS[walls], u_in=(0.08, 0.01), gbetaT=W.GBETA_T * 5, dir_theta=-0.4)
    f, orient = W.random_fields(nx, ny, rng_seed=7)
    for n in counts:
        out = []
        for passes in (False, True):
            s = L.Simulation(p, storage)
            s.init_fields(f, orient)
            s.set_profiling(passes)
            s.step(n)
            out.append(s.state())
        d = float(np.abs(out[0] - out[1]).max())
        assert d <= TOL[storage], (n, d)


# with 16-bit storage the steps that no graph holds run the passes, which round
# every wall value: the same bits as one step at a time
@pytest.mark.parametrize("storage", ["fp16", "bf16"])
@pytest.mark.parametrize("batch", [False, True])
def test_remainder_steps_keep_the_passes_rounding(storage, batch):
    from paper_2209_01444_gb300 import lbm as L

    p = W.thermosolutal_params(45, 38, bc=WALLS["open"], u_in=(0.08, 0.01), gbetaT=W.GBETA_T * 5)
    seeds = np.array([[20.0, 18.0, 5.0, 0.0]])
    out = []
    for calls in ((13,), (1,) * 13):
        if batch:
            s = L.Batch([p], storage=storage)
            s.init_seeds(0, seeds, -0.55, -0.3)
        else:
            s = L.Simulation(p, storage)
            s.init_seeds(seeds, -0.55, -0.3)
        for n in calls:
            s.step(n)
        out.append(s.fields(0) if batch else s.fields())
    for name in out[0]:
        assert np.array_equal(out[0][name], out[1][name]), name

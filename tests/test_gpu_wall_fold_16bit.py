"""16-bit storage inside a 16-step graph, where walls are updated by the next
step as it loads them (all walls up to 2^20 nodes, the columns on larger grids),
against profiled steps, which run the wall passes after every step.  The passes
round every wall value they store; a column that the next step updates is not
rounded.  A deviation near 1 rounds by 2^-12 in FP16 and 2^-9 in BF16; one such
rounding a step is allowed.  A wall cell taken from the wrong node is off by
O(0.1)."""
import numpy as np
import pytest

from paper_2209_01444_gb300 import workloads as W

pytestmark = pytest.mark.gpu

WALLS = {"open": ("inflow", "outflow", "symmetry", "symmetry"), "rows": ("periodic", "periodic", "noslip", "dirichlet"),
         "box": ("noslip", "dirichlet", "symmetry", "noslip")}
ROUNDING = {"fp16": 2.0 ** -12, "bf16": 2.0 ** -9}


@pytest.mark.parametrize("nx,ny,walls", [(4, 4, "box"), (33, 5, "open"), (34, 9, "rows"), (64, 6, "box"),
                                         (31, 7, "open"), (1040, 1032, "open")])
@pytest.mark.parametrize("storage", sorted(ROUNDING))
def test_graph_steps_against_the_passes(nx, ny, walls, storage):
    from paper_2209_01444_gb300 import lbm as L

    p = W.thermosolutal_params(nx, ny, bc=WALLS[walls], u_in=(0.08, 0.01), gbetaT=W.GBETA_T * 5, dir_theta=-0.4)
    f, orient = W.random_fields(nx, ny, rng_seed=7)
    out = []
    for passes in (False, True):
        s = L.Simulation(p, storage)
        s.init_fields(f, orient)
        s.set_profiling(passes)
        s.step(16)
        out.append(s.state())
    assert float(np.abs(out[0] - out[1]).max()) <= 16 * ROUNDING[storage]

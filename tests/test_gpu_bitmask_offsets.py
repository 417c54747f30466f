"""GPU: the bitmask grouping with 32-bit offsets gives what the memory grouping
gives, bit for bit, for every storage, collision, lattice and block edge, on a
ragged box with walls, an obstacle, an inlet and an outlet."""
import numpy as np
import pytest

from cases import make_grid

from paper_2503_07898_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("collision", ["bgk", "reg"])
@pytest.mark.parametrize("q", [19, 27])
@pytest.mark.parametrize("edge", [4, 8])
def test_bitmask_equals_memory_grouping(lbm, storage, collision, q, edge):
    nx, ny, nz = 53, 26, 30
    flags = np.zeros((nz, ny, nx), np.uint8)
    flags[:, 0] = flags[:, -1] = flags[0] = flags[-1] = 1
    flags[12:17, 10:15, 17:22] = 1
    flags[1:-1, 1:-1, 0] = 2 | (1 << 3)
    flags[1:-1, 1:-1, -1] = 3
    bc = np.zeros((4,) + flags.shape)
    bc[0][(flags & 7) == 2] = 0.03
    bc[3] = 1.0
    rho, u = wl.random_fields(flags.shape, seed=8, u_amp=0.03)
    out = []
    for schedule in ("disaggregated", "bitmask"):
        g = make_grid(lbm, "sparse", flags, bc, 0.56, collision, storage, schedule=schedule, block_edge=edge, lattice=q)
        lbm.lbm_init_equilibrium(g, 0, rho, u)
        lbm.lbm_step(g, 9)
        out.append(lbm.lbm_get_populations_f64(g, 0))
        lbm.lbm_grid_destroy(g)
    assert np.array_equal(out[0], out[1], equal_nan=True)

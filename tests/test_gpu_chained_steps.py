"""GPU: n steps in one call, whose launches overlap (programmatic dependent
launch) and hold both groups of the grid, against n calls with a wait after
each, bit for bit.

The single steps run the same kernels on the same inputs, so any difference is
a read of a value that the step before had not written yet.  Grids from less
than one CTA to several waves, with and without a boundary group; profiled
steps (a launch per group) agree as well.
"""
import numpy as np
import pytest

from cases import make_grid

from paper_2503_07898_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def state(lbm, g):
    import torch
    t = torch.empty(lbm.lbm_get_info(g)["population_bytes"][0], dtype=torch.uint8, device="cuda")
    lbm.lbm_get_populations(g, 0, t)
    return t


def compare(lbm, grids, n):
    import torch
    one, many, prof = grids
    lbm.lbm_step(one, n)
    for _ in range(n):
        lbm.lbm_step(many, 1)
        lbm.lbm_sync(many)
    lbm.lbm_profile(prof, 1)
    lbm.lbm_step(prof, n)
    lbm.lbm_profile(prof, 0)
    a, b, c = (state(lbm, g) for g in grids)
    assert torch.equal(a, b) and torch.equal(a, c)
    for g in grids:
        lbm.lbm_grid_destroy(g)


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("q", [19, 27])
@pytest.mark.parametrize("dims,lid", [((5, 3, 4), False), ((32, 32, 32), False), ((96, 70, 200), False),
                                      ((5, 4, 4), True), ((33, 31, 9), True), ((200, 96, 70), True)])
def test_dense(lbm, dims, lid, q, storage):
    grids = []
    for _ in range(3):
        if lid:
            flags, bc = wl.cavity(0, dims=dims)
            g = make_grid(lbm, "dense", flags, bc, 0.56, storage=storage, lattice=q)
        else:
            g = lbm.lbm_grid_create_dense(dims, lbm.physics(0.56, storage=storage, periodic=(1, 1, 1), lattice=q))
        rho, u = wl.random_fields(dims[::-1], seed=3, u_amp=0.03)
        lbm.lbm_init_equilibrium(g, 0, rho, u)
        grids.append(g)
    compare(lbm, grids, 31)


@pytest.mark.parametrize("storage", ["f32", "bf16"])
@pytest.mark.parametrize("edge", [4, 8])
@pytest.mark.parametrize("dims", [(24, 16, 16), (132, 66, 66)])
def test_sparse(lbm, dims, edge, storage):
    nx, ny, nz = dims
    flags = np.zeros((nz, ny, nx), np.uint8)
    flags[:, 0] = flags[:, -1] = flags[0] = flags[-1] = 1
    flags[1:-1, 1:-1, 0] = 2 | (1 << 3)
    flags[1:-1, 1:-1, -1] = 3
    flags[nz // 2, ny // 2, nx // 3] = 1
    bc = np.array([[0.03, 0, 0, 1] if f & 7 == 2 else [0, 0, 0, 1] for f in flags[flags & 6 == 2]], np.float32)
    grids = []
    for _ in range(3):
        g = lbm.lbm_grid_create_sparse(dims, edge, flags, lbm.physics(0.56, storage=storage))
        lbm.lbm_set_boundary(g, 0, None, bc)
        rho, u = wl.random_fields(flags.shape, seed=3, u_amp=0.03)
        lbm.lbm_init_equilibrium(g, 0, rho, u)
        grids.append(g)
    compare(lbm, grids, 21)

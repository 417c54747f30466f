"""GPU: lbm_profile(g, 2) records the launches that an unprofiled step makes: one
per step where both groups share it, with all updated voxels as its units."""
import numpy as np
import pytest

from cases import make_grid

from paper_2503_07898_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def profile(lbm, g, mode, n=5):
    lbm.lbm_step(g, 1)
    lbm.lbm_profile(g, mode)
    lbm.lbm_step(g, n)
    stats = lbm.lbm_profile_read(g)
    lbm.lbm_profile(g, 0)
    upd = lbm.lbm_get_info(g)["n_updated"][0]
    assert sum(s["units"] for s in stats.values()) == n * upd
    return {k: s["launches"] for k, s in stats.items()}


@pytest.mark.parametrize("dims,storage,q,want", [((40, 32, 24), "f32", 19, {"dense_step": 5}),
                                                 ((40, 32, 24), "bf16", 19, {"dense_step": 5}),
                                                 ((136, 128, 128), "f16", 19, {"dense_interior": 5, "dense_boundary": 5}),
                                                 ((136, 128, 128), "f32", 19, {"dense_step": 5}),
                                                 ((72, 64, 64), "f32", 27, {"dense_interior": 5, "dense_boundary": 5}),
                                                 ((64, 64, 64), "f32", 27, {"dense_step": 5})])
def test_dense(lbm, dims, storage, q, want):
    flags, bc = wl.cavity(0, dims=dims)
    g = make_grid(lbm, "dense", flags, bc, 0.6, storage=storage, lattice=q)
    lbm.lbm_init_equilibrium(g, 0, None, None)
    assert profile(lbm, g, 2) == want
    assert profile(lbm, g, 1) == {"dense_interior": 5, "dense_boundary": 5}
    lbm.lbm_grid_destroy(g)


@pytest.mark.parametrize("schedule,want", [("disaggregated", {"sparse_step": 5}),
                                           ("bitmask", {"sparse_interior_bitmask": 5, "sparse_boundary_bitmask": 5})])
@pytest.mark.parametrize("storage", ["f32", "f16"])
def test_sparse(lbm, storage, schedule, want):
    flags = np.zeros((24, 24, 40), np.uint8)
    flags[:, 0] = flags[:, -1] = flags[0] = flags[-1] = 1
    flags[1:-1, 1:-1, 0] = 2 | (1 << 3)
    flags[1:-1, 1:-1, -1] = 3
    bc = np.zeros((4,) + flags.shape)
    bc[3] = 1.0
    g = make_grid(lbm, "sparse", flags, bc, 0.6, storage=storage, schedule=schedule)
    lbm.lbm_init_equilibrium(g, 0, None, None)
    assert profile(lbm, g, 2) == want
    assert set(profile(lbm, g, 1)) == (set(want) if schedule == "bitmask" else {"sparse_interior", "sparse_boundary"})
    lbm.lbm_grid_destroy(g)

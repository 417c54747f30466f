"""GPU: FP32 batches of at most two work items per SM run an instantiation of their
own; around that line a batch gives what its grids give one by one, bit for bit."""
import numpy as np
import pytest

from paper_2503_07898_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def grid(lbm, kind, dims, collision, seed):
    flags = wl.random_obstacles(dims[::-1], seed=seed, solid_fraction=0.08)
    ph = lbm.physics(0.57, collision, "f32", (1, 1, 1))
    if kind == "dense":
        g = lbm.lbm_grid_create_dense(dims, ph)
        lbm.lbm_set_boundary(g, 0, flags)
    else:
        g = lbm.lbm_grid_create_sparse(dims, 8, flags, ph)
    rho, u = wl.random_fields(dims[::-1], seed=seed, u_amp=0.03)
    lbm.lbm_init_equilibrium(g, 0, rho, u)
    return g


@pytest.mark.parametrize("collision", ["bgk", "reg"])
@pytest.mark.parametrize("members", [[("dense", (16, 8, 8))], [("sparse", (24, 16, 16)), ("dense", (19, 7, 33))],
                                     [("dense", (76, 64, 32))],                                # 304 items
                                     [("dense", (77, 64, 32))],                                # 308
                                     [("sparse", (64, 64, 32)), ("dense", (32, 32, 24))],      # 304
                                     [("sparse", (64, 64, 32)), ("dense", (33, 32, 24))]])     # 306
def test_batch_equals_single_grids(lbm, members, collision):
    batch = [grid(lbm, k, d, collision, 11 + i) for i, (k, d) in enumerate(members)]
    alone = [grid(lbm, k, d, collision, 11 + i) for i, (k, d) in enumerate(members)]
    b = lbm.lbm_batch_create(batch)
    lbm.lbm_batch_step(b, 11)
    for (kind, _), g, h in zip(members, batch, alone):
        lbm.lbm_step(h, 11)
        f, ref = lbm.lbm_get_populations_f64(g, 0), lbm.lbm_get_populations_f64(h, 0)
        ok = np.isfinite(ref)
        assert np.array_equal(np.isfinite(f), ok)
        assert np.array_equal(f[ok], ref[ok])
    lbm.lbm_batch_destroy(b)
    for g in batch + alone:
        lbm.lbm_grid_destroy(g)

"""GPU: the closure dataset works in the population buffer that the next step
overwrites; the grid must not show it.  Steps after a dataset call, and walls
set after it, give what they give without the call, bit for bit; filters
wider than eight voxels take the compensated sums (tolerances as in
test_gpu_closure_kernels.py: a few 2^-24 of the populations' size for the
features, 1e-3 of the largest target)."""
import numpy as np
import pytest

from oracle import closure as ocl
from paper_2503_07898_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def make(lbm, dims, storage, r):
    rho, u = wl.turbulence(0, seed=4 + r, u_rms=0.03, kmax=2, dims=dims)
    g = lbm.lbm_grid_create_dense(dims, lbm.physics(0.52, storage=storage, periodic=(1, 1, 1)))
    lbm.lbm_init_equilibrium(g, 0, rho, u)
    return g


def dataset(lbm, g, dims, r):
    import torch
    nc = int(np.prod(dims)) // r ** 3
    feats, targ = torch.empty(nc, 16, device="cuda"), torch.empty(nc, device="cuda")
    lbm.lbm_closure_dataset(g, r, 0.5 + 0.02 / r, feats, targ)
    return feats.cpu().numpy(), targ.cpu().numpy()


def state(lbm, g):
    import torch
    t = torch.empty(lbm.lbm_get_info(g)["population_bytes"][0], dtype=torch.uint8, device="cuda")
    lbm.lbm_get_populations(g, 0, t)
    return t


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("r", [1, 2])
def test_dataset_leaves_the_grid_alone(lbm, r, storage):
    import torch
    dims = (24, 16, 12)
    a, b = make(lbm, dims, storage, r), make(lbm, dims, storage, r)
    for n in (1, 2):
        dataset(lbm, a, dims, r)
        assert torch.equal(state(lbm, a), state(lbm, b))
        lbm.lbm_step(a, n)
        lbm.lbm_step(b, n)
        assert torch.equal(state(lbm, a), state(lbm, b))


@pytest.mark.parametrize("storage", ["f32", "bf16"])
def test_walls_after_a_dataset(lbm, storage):
    """Solid voxels keep the buffers' initial zeros."""
    import torch
    dims = (24, 16, 12)
    flags = np.zeros(dims[::-1], np.uint8)
    flags[3:6, 4:9, 5:20] = 1
    a, b = make(lbm, dims, storage, 2), make(lbm, dims, storage, 2)
    dataset(lbm, a, dims, 2)
    for g in (a, b):
        lbm.lbm_set_boundary(g, 0, flags, None)
        lbm.lbm_step(g, 1)
    assert torch.equal(state(lbm, a), state(lbm, b))


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("r,dims", [(8, (24, 8, 16)), (9, (27, 18, 9)), (16, (32, 16, 32))])
def test_wide_filters(lbm, r, dims, storage):
    g = make(lbm, dims, storage, r)
    lbm.lbm_step(g, 3)
    f = lbm.lbm_get_populations_f64(g, 0)
    F, T = dataset(lbm, g, dims, r)
    ref = ocl.features(ocl.coarse_pulled(f, r), 0.5 + 0.02 / r).reshape(-1, 16)
    assert np.all(np.abs(F - ref) <= 1e-5 * np.abs(ref).max(axis=0) + 2e-6)
    want = ocl.eddy_target(f, r, 0.5 + 0.02 / r).ravel()
    assert np.abs(T - want).max() <= 1e-3 * np.abs(want).max()

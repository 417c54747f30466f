"""GPU: closure datasets of states outside the windows of the exact sums
(densities far from one, infinite populations), against the oracle and against the
rules of the FP64 form.

Tolerances.  Feature 0 is an FP32 sum of 19 filtered populations s (of one sign
for these densities), each rounded to FP32 once: 19 x 2^-24 of it, taken as
20 x 2^-24.  The other features are moments divided by rho / 3: rounding of s,
of a sum of 19 and of the subtractions gives at most 37 x 2^-24 = 2.2e-6 each,
three times that in the norm: 8e-6, plus 1e-5 of the largest value for the
products.  Targets: as in test_gpu_closure_kernels.py, 1e-3 of the largest."""
import numpy as np
import pytest

from oracle import closure as ocl
from paper_2503_07898_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def dataset(lbm, g, dims, r, tau):
    import torch
    nc = int(np.prod(dims)) // r ** 3
    feats, targ = torch.full((nc, 16), -7.0, device="cuda"), torch.full((nc,), -7.0, device="cuda")
    lbm.lbm_closure_dataset(g, r, tau, feats, targ)
    return feats.cpu().numpy(), targ.cpu().numpy()


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("r,dims", [(2, (12, 10, 8)), (3, (12, 9, 15)), (4, (16, 12, 8)), (5, (15, 20, 10)),
                                    (8, (24, 16, 16)), (17, (51, 34, 17))])
@pytest.mark.parametrize("scale", [10.0, 40.0])
def test_dense_fluids(lbm, storage, r, dims, scale):
    rho, u = wl.turbulence(0, seed=31 + r, u_rms=0.03, kmax=2, dims=dims)
    g = lbm.lbm_grid_create_dense(dims, lbm.physics(0.52, storage=storage, periodic=(1, 1, 1)))
    lbm.lbm_init_equilibrium(g, 0, scale * rho, u)
    f = lbm.lbm_get_populations_f64(g, 0)
    tau = 0.5 + 0.02 / r
    F, T = dataset(lbm, g, dims, r, tau)
    lbm.lbm_grid_destroy(g)
    ref = ocl.features(ocl.coarse_pulled(f, r), tau).reshape(-1, 16)
    assert np.all(np.abs(F[:, 0] - ref[:, 0]) <= 20 * 2.0 ** -24 * np.abs(ref[:, 0]))
    assert np.all(np.abs(F - ref)[:, 1:] <= 1e-5 * np.abs(ref[:, 1:]).max(axis=0) + 8e-6)
    want = ocl.eddy_target(f, r, tau).ravel()
    assert np.abs(T - want).max() <= 1e-3 * np.abs(want).max()


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("r,dims", [(3, (12, 9, 6)), (4, (8, 12, 16)), (5, (15, 10, 20)), (8, (16, 24, 8))])
@pytest.mark.parametrize("rho0", [0.03, 1.9, 10.0, 40.0])
def test_uniform_fluids(lbm, storage, r, dims, rho0):
    """Equal populations: every addition rounds the same way."""
    g = lbm.lbm_grid_create_dense(dims, lbm.physics(0.52, storage=storage, periodic=(1, 1, 1)))
    lbm.lbm_init_equilibrium(g, 0, np.full(dims[::-1], rho0), np.zeros((3,) + dims[::-1]))
    f = lbm.lbm_get_populations_f64(g, 0)
    F, T = dataset(lbm, g, dims, r, 0.51)
    lbm.lbm_grid_destroy(g)
    drho = float((f[:, 0, 0, 0]).sum()) - 1.0
    assert np.all(np.abs(F[:, 0] - drho) <= 20 * 2.0 ** -24 * abs(drho))
    assert np.all(T == 0.0)


@pytest.mark.parametrize("r", [2, 4])
def test_infinite_population(lbm, r):
    """An infinite rest population is an infinite density of its own coarse
    voxel and reaches no other one's features."""
    dims = (16, 16, 8)
    rho, u = wl.turbulence(0, seed=3, u_rms=0.03, kmax=2, dims=dims)
    g = lbm.lbm_grid_create_dense(dims, lbm.physics(0.52, periodic=(1, 1, 1)))
    lbm.lbm_init_equilibrium(g, 0, rho, u)
    clean, _ = dataset(lbm, g, dims, r, 0.51)
    f = np.empty(19 * rho.size, np.float32)
    lbm.lbm_get_populations(g, 0, f)
    f[5 + 16 * (6 + 16 * 3)] = np.inf  # population 0 of voxel (5, 6, 3)
    lbm.lbm_set_populations(g, 0, f)
    F, _ = dataset(lbm, g, dims, r, 0.51)
    lbm.lbm_grid_destroy(g)
    hit = 5 // r + (16 // r) * (6 // r + (16 // r) * (3 // r))
    assert F[hit, 0] == np.inf
    rest = np.arange(len(F)) != hit
    assert np.array_equal(F[rest], clean[rest])


@pytest.mark.parametrize("tau", [0.5005, 0.501, 0.75])
def test_target_bounds_without_gradients(lbm, tau):
    """No velocity gradient: the target is 0 brought into its bounds, whose lower
    one is positive for tau < 0.501."""
    dims = (8, 12, 16)
    g = lbm.lbm_grid_create_dense(dims, lbm.physics(0.52, periodic=(1, 1, 1)))
    lbm.lbm_init_equilibrium(g, 0, np.ones(dims[::-1]), np.zeros((3,) + dims[::-1]))
    f = lbm.lbm_get_populations_f64(g, 0)
    _, T = dataset(lbm, g, dims, 2, tau)
    lbm.lbm_grid_destroy(g)
    want = ocl.eddy_target(f, 2, float(np.float32(tau))).ravel()
    assert np.array_equal(T, want.astype(np.float32))

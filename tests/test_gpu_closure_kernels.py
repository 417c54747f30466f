"""GPU: the fused training kernels, the column statistics and the dataset
kernels at the sizes where their tiling can go wrong: batches around the
32-sample tile and beyond one tile per CTA, sample counts around the CTA rows,
unaligned feature arrays, box filters of odd width on odd boxes.

Tolerances: gradients and one Adam step as in test_gpu_closure.py (FP32
against FP64, norm-wise 1e-5).  Dataset features are FP32 moments of FP32
filtered populations: a few 2^-24 of the populations' size, scaled by 3, so
2e-6 absolute plus 1e-5 relative; the target is a ratio of differences a
thousand times smaller than the stored FP32 means (2^-24 x 1e3), so 1e-3 of
its largest value, as in test_gpu_closure.py.
"""
import numpy as np
import pytest

from oracle import closure as ocl
from oracle import lattice as OL
from paper_2503_07898_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def cuda(a, dtype=np.float32):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a, dtype=dtype)).cuda()


def weights(seed):
    rng = np.random.default_rng(seed)
    return np.concatenate([rng.standard_normal(1024) * np.sqrt(2 / 16), 0.1 * rng.standard_normal(64),
                           rng.standard_normal(4096) * np.sqrt(2 / 64), 0.1 * rng.standard_normal(64),
                           rng.standard_normal(64) / 8, np.zeros(1)]).astype(np.float32)


@pytest.mark.parametrize("batch", [1, 31, 32, 33, 304 * 32, 304 * 32 + 5])
def test_gradient_over_tile_edges(lbm, batch):
    import torch
    rng = np.random.default_rng(batch)
    n = 500
    X = rng.standard_normal((n, 16)).astype(np.float32)
    t = rng.standard_normal(n).astype(np.float32)
    idx = rng.integers(0, n, batch).astype(np.int32)
    th = weights(batch + 1)
    g = torch.full((5313,), float("nan"), device="cuda")
    loss = torch.full((1,), float("nan"), device="cuda")
    lbm.lbm_closure_grad(cuda(th), cuda(X), cuda(t), cuda(idx, np.int32), g, loss)
    ref_loss, ref = ocl.loss_and_grad(th.astype(np.float64), X[idx].astype(np.float64), t[idx].astype(np.float64))
    got = g.cpu().numpy().astype(np.float64)
    assert np.linalg.norm(got - ref) <= 1e-5 * np.linalg.norm(ref)
    assert abs(loss.item() - ref_loss) <= 1e-5 * ref_loss


@pytest.mark.parametrize("n,shift", [(1, 0), (63, 1), (64, 0), (65, 2), (304 * 64 + 3, 1), (50001, 0)])
def test_statistics_and_one_step(lbm, n, shift):
    """One Adam step; the features start `shift` floats into their buffer, one
    column has a mean 1e5 times its deviation and one is constant."""
    import torch
    rng = np.random.default_rng(n)
    X = rng.standard_normal((n, 16)) * np.logspace(-4, 0, 16) + rng.standard_normal(16)
    X[:, 3] = 1000.0 + 0.01 * rng.standard_normal(n)
    X[:, 15] = 0.501
    X = X.astype(np.float32)
    t = (0.01 * rng.standard_normal(n) + 0.003).astype(np.float32)
    buf = torch.zeros(16 * n + shift, device="cuda")
    buf[shift:] = cuda(X).view(-1)
    th0 = weights(n + 1)
    th = cuda(th0)
    loss = lbm.lbm_closure_train(buf[shift:].view(n, 16), cuda(t), 1, 96, 1e-3, 5, th)
    ref, ref_loss = ocl.train(X.astype(np.float64), t.astype(np.float64), th0.astype(np.float64), 1, 96, 1e-3, 5)
    err = th.cpu().numpy() - ref
    # (X - mu) / sd of the column with the large mean: its mean rounded to
    # FP32 moves it by up to 2^-25 1000 / 0.01 = 3e-3 deviations
    tol = 1e-5 if n == 1 else 5e-3
    for a, b in ((0, 1024), (1088, 5184), (5248, 5312)):
        assert np.linalg.norm(err[a:b]) <= tol * np.linalg.norm(ref[a:b])
    assert abs(loss - ref_loss) <= tol * ref_loss + 1e-12


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("r,dims", [(1, (9, 7, 5)), (2, (18, 6, 10)), (3, (21, 9, 6)), (5, (15, 35, 10))])
def test_dataset_over_filters(lbm, r, dims, storage):
    import torch
    tau_f = 0.52
    tau_c = 0.5 + (tau_f - 0.5) / r
    rho, u = wl.turbulence(0, seed=9 + r, u_rms=0.03, kmax=2, dims=dims)
    g = lbm.lbm_grid_create_dense(dims, lbm.physics(tau_f, storage=storage, periodic=(1, 1, 1)))
    lbm.lbm_init_equilibrium(g, 0, rho, u)
    lbm.lbm_step(g, 3)
    f = lbm.lbm_get_populations_f64(g, 0)
    nc = int(np.prod(dims)) // r ** 3
    buf = torch.empty(nc * 16 + 1, device="cuda")
    for shift in (0, 1):  # aligned and unaligned feature rows
        feats, targ = buf[shift:shift + nc * 16], torch.empty(nc, device="cuda")
        lbm.lbm_closure_dataset(g, r, tau_c, feats, targ)
        F_ref = ocl.features(ocl.coarse_pulled(f, r), tau_c).reshape(-1, 16)
        F = feats.view(nc, 16).cpu().numpy()
        assert np.all(np.abs(F - F_ref) <= 1e-5 * np.abs(F_ref).max(axis=0) + 2e-6)
        if r == 1:
            continue  # no sub-filter stress: the target is a ratio of rounding errors
        T_ref = ocl.eddy_target(f, r, tau_c).ravel()
        T = targ.cpu().numpy()
        assert np.abs(T - T_ref).max() <= 1e-3 * np.abs(T_ref).max()

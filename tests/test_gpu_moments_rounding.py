"""GPU: rho and u read out are the exact sums of the stored populations and
their correctly rounded quotients: sums of 19 or 27 stored values in FP64 are
exact, in any order, for FP32 populations in [2^-11, 2) and for 16-bit ones
below 1/2, so numpy gives both to the last bit and no difference is allowed."""
import numpy as np
import pytest

from oracle import lattice as OL

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("q", [19, 27])
@pytest.mark.parametrize("rho0,u_amp", [(1.0, 0.1), (1.7, 1e-3), (0.35, 0.2), (0.08, 0.15)])
def test_moments_are_correctly_rounded(lbm, storage, q, rho0, u_amp):
    import torch
    if storage == "f32" and rho0 < 0.3:
        rho0 = 0.4  # FP32 corners of D3Q27 would leave the window
    dims = (72, 40, 33)
    n = int(np.prod(dims))
    rng = np.random.default_rng(int(100 * rho0) + q)
    rho = rho0 * (1.0 + 0.01 * rng.uniform(-1, 1, dims[::-1]))
    u = u_amp * rng.uniform(-1, 1, (3,) + dims[::-1])
    g = lbm.lbm_grid_create_dense(dims, lbm.physics(0.6, storage=storage, periodic=(1, 1, 1), lattice=q))
    lbm.lbm_init_equilibrium(g, 0, rho, u)
    raw = torch.empty(q * n, dtype={"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}[storage],
                      device="cuda")
    lbm.lbm_get_populations(g, 0, raw)
    r, v = lbm.lbm_get_moments(g, 0)
    lbm.lbm_grid_destroy(g)
    f = raw.double().cpu().numpy().reshape((q,) + dims[::-1])
    C = (OL.D3Q19.C if q == 19 else OL.D3Q27.C).astype(np.float64)
    want = f.sum(axis=0) + (0.0 if storage == "f32" else 1.0)
    j = np.stack([sum(C[i, a] * f[i] for i in range(q) if C[i, a]) for a in range(3)])
    ok = np.ones_like(want, bool)
    if storage != "f32":
        ok = ((f == 0.0) | (np.abs(f) >= 2.0 ** -33)).all(axis=0)  # BF16 values with bits below 2^-40
    assert ok.mean() > 0.99
    assert np.array_equal(r[ok], want[ok])
    assert np.array_equal(v[:, ok], (j / want)[:, ok])

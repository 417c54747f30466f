"""GPU: initial state, moments and conservation sums inside and outside the
windows of their exact forms, dense and 8^3 / 4^3 sparse, both lattices.

Tolerances.  rho is one rounding of the exact sum, the reference an FP64 sum
of 27 terms: 27 2^-53 of the sum of magnitudes.  u = j / rho adds the same
absolute error of j and two roundings: 30 2^-53 (sum |f|) / |rho| (1 + |u|).
Conservation sums n voxels: n such errors.  The initial state is one rounding
of an evaluation whose relative error is below 2^-43 of f; the FP64 reference
is as good, so FP32 values are at most one ulp apart (near-ties) and 16-bit
ones one unit in the last place plus 2^-43.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def lattice(q):
    c = np.array([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
                  (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1),
                  (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1),
                  (1, 1, 1), (-1, -1, -1), (1, 1, -1), (-1, -1, 1), (1, -1, 1), (-1, 1, -1),
                  (-1, 1, 1), (1, -1, -1)], float)[:q]
    n = np.abs(c).sum(1).astype(int)
    per = {19: (1 / 3, 1 / 18, 1 / 36), 27: (8 / 27, 2 / 27, 1 / 54, 1 / 216)}[q]
    return c, np.array([per[k] for k in n])


def grid(lbm, kind, dims, storage, q):
    ph = lbm.physics(0.6, storage=storage, periodic=(1, 1, 1), lattice=q)
    if kind == "dense":
        return lbm.lbm_grid_create_dense(dims, ph)
    return lbm.lbm_grid_create_sparse(dims, int(kind[-1]), np.zeros(dims[::-1], np.uint8), ph)


def values(rng, n, w, storage):
    """Populations (q, n) as the storage holds them, absolute in FP64: ordinary
    voxels, voxels at the edges of the exact windows and outside them."""
    q = len(w)
    f = w[:, None] * (1 + 0.2 * rng.uniform(-1, 1, (q, n)))
    kind = rng.integers(0, 8, n)
    i = rng.integers(0, q, n)
    f[i[kind == 1], np.flatnonzero(kind == 1)] = 2.0 ** -11
    f[i[kind == 2], np.flatnonzero(kind == 2)] = np.nextafter(np.float32(2.0 ** -11), np.float32(0))
    f[i[kind == 3], np.flatnonzero(kind == 3)] = np.nextafter(np.float32(2), np.float32(0))
    f[i[kind == 4], np.flatnonzero(kind == 4)] = 3.25
    f[i[kind == 5], np.flatnonzero(kind == 5)] = -0.01
    f[:, kind == 6] = w[:, None] * (1 + rng.uniform(-1, 1, (q, (kind == 6).sum())) * 1e-12)
    f[:, kind == 7] *= 70
    if storage == "f32":
        s = f.astype(np.float32)
        return s, s.astype(np.float64)
    import torch
    t = torch.from_numpy(f - w[:, None]).to(torch.float16 if storage == "f16" else torch.bfloat16)
    return t, t.double().numpy() + w[:, None]


@pytest.mark.parametrize("q", [19, 27])
@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("kind,dims", [("dense", (1, 1, 1)), ("dense", (37, 5, 9)), ("sparse8", (24, 8, 16)),
                                       ("sparse4", (12, 8, 4))])
def test_moments_and_sums(lbm, kind, dims, storage, q):
    import torch
    c, w = lattice(q)
    n = int(np.prod(dims))
    rng = np.random.default_rng(n + q)
    raw, f = values(rng, n, w, storage)
    g = grid(lbm, kind, dims, storage, q)
    if kind == "dense":
        buf = raw
        order = np.arange(n)
    else:
        # storage slot of each voxel from an initial state whose density is its id
        e3 = int(kind[-1]) ** 3
        probe = grid(lbm, kind, dims, "f32", q)
        lbm.lbm_init_equilibrium(probe, 0, (np.arange(n, dtype=np.float64) + 1).reshape(dims[::-1]),
                                 np.zeros((3,) + dims[::-1]))
        p = np.empty(n * q, np.float32)
        lbm.lbm_get_populations(probe, 0, p)
        order = np.rint(p.reshape(-1, q, e3)[:, 0] / w[0]).astype(int).ravel() - 1
        assert sorted(order) == list(range(n))
        buf = raw[:, order].reshape(q, -1, e3)
        buf = buf.permute(1, 0, 2) if storage != "f32" else buf.transpose(1, 0, 2)
    t = torch.from_numpy(np.ascontiguousarray(buf)).cuda() if storage == "f32" else buf.contiguous().cuda()
    lbm.lbm_set_populations(g, 0, t)
    rho = torch.empty(dims[::-1], dtype=torch.float64, device="cuda")
    u = torch.empty((3,) + dims[::-1], dtype=torch.float64, device="cuda")
    lbm.lbm_get_moments(g, 0, rho, u)
    rho, u = rho.cpu().numpy().ravel(), u.cpu().numpy().reshape(3, n)
    m, j, mag = f.sum(0), c.T @ f, np.abs(f).sum(0) + 1.0
    assert np.all(np.abs(rho - m) <= 30 * 2.0 ** -53 * mag)
    assert np.all(np.abs(u - j / m) <= 32 * 2.0 ** -53 * mag / np.abs(m) * (1 + np.abs(j / m)))
    sums = lbm.lbm_conservation(g)
    ref = np.concatenate([[m.sum()], j.sum(1)])
    assert np.all(np.abs(np.asarray(sums) - ref) <= 64 * 2.0 ** -53 * mag.sum())


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_voxel(lbm, bad):
    import torch
    g = grid(lbm, "dense", (5, 4, 3), "f32", 19)
    _, w = lattice(19)
    f = np.tile(w[:, None], (1, 60)).astype(np.float32)
    f[4, 17] = bad
    lbm.lbm_set_populations(g, 0, torch.from_numpy(f).cuda())
    rho = torch.empty(60, dtype=torch.float64, device="cuda")
    u = torch.empty(3, 60, dtype=torch.float64, device="cuda")
    lbm.lbm_get_moments(g, 0, rho.view(3, 4, 5), u.view(3, 3, 4, 5))
    rho = rho.cpu().numpy()
    assert (np.isnan(rho[17]) if np.isnan(bad) else np.isposinf(rho[17]))
    assert np.all(np.isfinite(np.delete(rho, 17)))
    with pytest.raises(lbm.LbmError, match="non-finite"):
        lbm.lbm_conservation(g)


@pytest.mark.parametrize("q", [19, 27])
@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("kind,dims", [("dense", (41, 7, 6)), ("sparse8", (24, 8, 16))])
def test_initial_state(lbm, kind, dims, storage, q):
    import torch
    c, w = lattice(q)
    n = int(np.prod(dims))
    rng = np.random.default_rng(q)
    rho = rng.uniform(0.9, 1.1, n)
    u = rng.uniform(-0.2, 0.2, (3, n))
    k = rng.integers(0, 10, n)
    u[:, k == 1] = 0.0
    u[0, k == 2] = 0.2499999999
    u[1, k == 3] = -0.25
    u[2, k == 4] = 0.4
    u[:, k == 5] *= 1e-20
    u[0, k == 6] = 1e-310
    rho[k == 7] = rng.uniform(200, 300, (k == 7).sum())
    rho[k == 8] = 1.0
    u[:, k == 8] = 0.0
    rho[k == 9] = 2.0 ** -9
    g = grid(lbm, kind, dims, storage, q)
    lbm.lbm_init_equilibrium(g, 0, rho.reshape(dims[::-1]), u.reshape((3,) + dims[::-1]))
    got = np.asarray(lbm.lbm_get_populations_f64(g, 0)).reshape(q, n)
    cu = c @ u
    ref = w[:, None] * rho * (1 + 3 * cu + 4.5 * cu ** 2 - 1.5 * (u ** 2).sum(0))
    if storage == "f32":
        near = ref.astype(np.float32).astype(np.float64)
        assert np.all(np.abs(got - near) <= np.spacing(np.abs(near).astype(np.float32)))
        assert np.mean(got != near) <= 1e-3
    else:
        t = torch.float16 if storage == "f16" else torch.bfloat16
        s = torch.from_numpy(ref - w[:, None])
        near = s.to(t).double().numpy()
        # one ulp of the stored value, the smallest spacing of FP16 and the
        # evaluation's own error
        tol = np.abs(near) * (2.0 ** -10 if storage == "f16" else 2.0 ** -7) + \
            (2.0 ** -24 if storage == "f16" else 0.0) + 2.0 ** -43 * np.abs(ref)
        assert np.all(np.abs(got - w[:, None] - near) <= tol + 2.0 ** -52 * np.abs(got))
        assert np.mean(np.abs(got - w[:, None] - near) > 2.0 ** -43 * np.abs(ref) + 1e-16) <= 1e-3

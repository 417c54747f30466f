"""Performance cases: what a user of the library has it do, through the public
binding, over the range of sizes, layouts, storages and options it is used with.

A case is a dict of plain values; its "kind" selects the path:
  dense     lbm_step on a dense grid, then the stored populations
  sparse    lbm_step on an 8^3 block-sparse sphere channel, then the populations
  multires  lbm_step on a three-level grid (optionally with the learned
            closure), then the populations of every level
  batch     lbm_batch_step over independent grids, then their populations
  learn     lbm_closure_dataset on a checkpoint, then lbm_closure_train on it
  readout   lbm_init_equilibrium, lbm_get_moments, lbm_conservation

`exact` evaluates the same path in plain 64-bit torch.
"""
import functools
import math

import numpy as np
import torch

from paper_2503_07898_gb300 import binding as lbm

DEV = "cuda" if torch.cuda.is_available() else "cpu"
BYTES = {"f32": 4, "f16": 2, "bf16": 2}
DTYPE = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
FLUID, SOLID, VELOCITY, PRESSURE, OUTSIDE = 0, 1, 2, 3, 7

# the library's velocity order: rest, 6 axes, 12 edges, 8 corners
C = np.array([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
              (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1),
              (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1),
              (1, 1, 1), (-1, -1, -1), (1, 1, -1), (-1, -1, 1), (1, -1, 1), (-1, 1, -1),
              (-1, 1, 1), (1, -1, -1)])


def weights(q):
    per = {19: (1 / 3, 1 / 18, 1 / 36), 27: (8 / 27, 2 / 27, 1 / 54, 1 / 216)}[q]
    return [per[int(np.abs(C[i]).sum())] for i in range(q)]


def opposite(i):
    return 0 if i == 0 else (i + 1 if i % 2 else i - 1)


# ------------------------------------------------------------------- cases

def listed():
    return [
        # the smallest: the 32^3 periodic Taylor-Green-sized box, one call of
        # 100 steps; launches and latency count, the state fits in L2
        dict(name="box32_f32", kind="dense", nx=32, ny=32, nz=32, walls="periodic", storage="f32",
             collision="bgk", q=19, tau=0.6, steps=100),
        # the headline: 256^3 lid-driven cavity in FP32 and in FP16 storage
        dict(name="cavity256_f32", kind="dense", nx=256, ny=256, nz=256, walls="cavity",
             storage="f32", collision="bgk", q=19, tau=0.515, steps=20),
        dict(name="cavity256_f16", kind="dense", nx=256, ny=256, nz=256, walls="cavity",
             storage="f16", collision="bgk", q=19, tau=0.515, steps=20),
        # odd, ragged box with obstacles, periodic along x, BF16 storage,
        # regularized collision: a porous duct
        dict(name="duct_bf16_reg", kind="dense", nx=181, ny=93, nz=77, walls="duct",
             storage="bf16", collision="reg", q=19, tau=0.56, steps=40),
        # the 512x256x256 flow past a sphere in a channel on 8^3 blocks
        dict(name="sphere_f32", kind="sparse", nx=512, ny=256, nz=256, storage="f32",
             collision="bgk", q=19, tau=0.52, steps=20),
        dict(name="sphere_f16", kind="sparse", nx=512, ny=256, nz=256, storage="f16",
             collision="bgk", q=19, tau=0.52, steps=20),
        # the same channel at half size (a ragged box) with D3Q27 and the
        # regularized collision
        dict(name="sphere_q27_reg", kind="sparse", nx=260, ny=132, nz=132, storage="f32",
             collision="reg", q=27, tau=0.52, steps=20),
        # 256^3 three-level decaying turbulence: FP16 storage, and FP32 with
        # the learned closure on the coarser levels; one step is one coarsest
        # step, four finest ones
        dict(name="levels256_f16", kind="multires", nx=256, ny=256, nz=256, storage="f16",
             collision="bgk", q=19, tau=0.52, steps=8, closure=False),
        dict(name="levels256_closure", kind="multires", nx=256, ny=256, nz=256, storage="f32",
             collision="bgk", q=19, tau=0.504, steps=8, closure=True),
        # serving: 16 independent grids of mixed size and kind, one call
        dict(name="batch16_f16", kind="batch", n=16, lo=32, hi=160, storage="f16",
             collision="bgk", steps=50),
        # training data from a 256^3 checkpoint, then 20 minibatches of 4096:
        # the start of a training run (over hundreds of Adam steps the last
        # bits of the gradients grow until runs can no longer be compared)
        dict(name="learn256", kind="learn", nx=256, ny=256, nz=256, r=2, storage="f32",
             tau=0.508, steps=20, batch=4096),
        # set up a 256^3 run from given fields, read density and velocity
        # back, check conservation
        dict(name="readout256_f32", kind="readout", nx=256, ny=256, nz=256, storage="f32", q=19),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["dense", "dense", "dense", "sparse", "sparse", "multires", "multires", "batch", "learn", "readout"])
    storage = rng.choice(["f32", "f16", "bf16"])
    collision = rng.choice(["bgk", "bgk", "reg"])
    q = rng.choice([19, 19, 19, 27])
    tau = round(rng.uniform(0.51, 0.8), 3)
    if kind == "dense":
        n = [_log(rng, 16, 256) for _ in range(3)]
        return dict(kind=kind, nx=n[0], ny=n[1], nz=n[2], walls=rng.choice(["periodic", "cavity", "duct"]),
                    storage=storage, collision=collision, q=q, tau=tau,
                    steps=max(5, min(100, 20 * 256 ** 3 // (n[0] * n[1] * n[2]))))
    if kind == "sparse":
        n = _log(rng, 60, 256)
        return dict(kind=kind, nx=n + _log(rng, 20, 200), ny=n, nz=n, storage=storage,
                    collision=collision, q=q, tau=tau, steps=rng.randint(5, 20))
    if kind == "multires":
        n = [32 * rng.randint(1, 8) for _ in range(2)]
        return dict(kind=kind, nx=n[0], ny=n[1], nz=256, storage=storage, collision=collision, q=19,
                    tau=tau, steps=rng.randint(2, 8), closure=rng.choice([False, False, True]))
    if kind == "batch":
        return dict(kind=kind, n=rng.randint(1, 16), lo=32, hi=rng.choice([64, 96, 128, 160]),
                    storage=storage, collision=collision, steps=rng.randint(5, 50))
    if kind == "learn":
        r = rng.choice([2, 3, 4])
        n = [r * (_log(rng, 24, 240) // r) for _ in range(3)]
        return dict(kind=kind, nx=n[0], ny=n[1], nz=n[2], r=r, storage=storage, tau=0.508,
                    steps=rng.randint(5, 20), batch=_log(rng, 512, 8192))
    n = [_log(rng, 16, 256) for _ in range(3)]
    return dict(kind="readout", nx=n[0], ny=n[1], nz=n[2], storage=storage, q=q)


# ------------------------------------------------------------------- inputs

def _gen(seed):
    return torch.Generator().manual_seed(seed)


def fields(dims, seed, u_rms=0.03, modes=8, kmax=6):
    """Smooth seeded density and velocity (float64, on the GPU): the sum of a
    few low-wavenumber Fourier modes, periodic in the box."""
    nx, ny, nz = dims
    rnd = torch.rand(modes, 4, 3, generator=_gen(seed), dtype=torch.float64).tolist()
    ax = [torch.arange(n, device=DEV, dtype=torch.float64) * (2 * math.pi / n) for n in (nx, ny, nz)]
    out = torch.zeros(4, nz, ny, nx, device=DEV, dtype=torch.float64)
    for m in rnd:
        for a in range(4):
            k = [1 + int(m[(a + b) % 4][b] * kmax) for b in range(3)]
            s = [torch.sin(k[b] * ax[b] + 2 * math.pi * m[a][b]) for b in range(3)]
            out[a] += s[2][:, None, None] * s[1][None, :, None] * s[0][None, None, :]
    out *= u_rms * math.sqrt(8.0 / modes)
    return 1.0 + 0.1 * out[0], out[1:].contiguous()


def equilibrium(rho, u, q):
    usq = 1.5 * (u * u).sum(0)
    w = weights(q)
    f = torch.empty((q,) + tuple(rho.shape), dtype=rho.dtype, device=rho.device)
    for i in range(q):
        cu = sum(float(C[i][a]) * u[a] for a in range(3) if C[i][a]) if i else torch.zeros_like(rho)
        f[i] = w[i] * rho * (1 + 3 * cu + 4.5 * cu * cu - usq)
    return f


def stored(f, storage):
    """Populations (float64, absolute) in the storage format."""
    if storage == "f32":
        return f.float()
    w = torch.tensor(weights(f.shape[0]), dtype=f.dtype, device=f.device).view(-1, 1, 1, 1)
    return (f - w).to(DTYPE[storage])


def absolute(s, q):
    """Inverse of stored()."""
    if s.dtype == torch.float32:
        return s.double()
    return s.double() + torch.tensor(weights(q), dtype=torch.float64, device=s.device).view(-1, 1, 1, 1)


def checkpoint(dims, seed, tau, storage):
    """D3Q19 post-collision state of a periodic flow: equilibrium plus the
    viscous part -tau w_i rho 3 Q_i : grad u (1 - 1 / tau), as a run stores it."""
    rho, u = fields(dims, seed, kmax=max(1, min(dims) // 8))
    f = equilibrium(rho, u, 19)
    w = weights(19)
    for b in range(3):
        for a in range(3):
            g = 0.5 * (torch.roll(u[b], -1, 2 - a) - torch.roll(u[b], 1, 2 - a)) * rho
            for i in range(19):
                coef = float(C[i][a] * C[i][b]) - (1 / 3 if a == b else 0.0)
                if coef:
                    f[i] += (1 - tau) * 3 * w[i] * coef * g
    return stored(f, storage).contiguous()


def _spheres(flags, fraction, rng):
    nz, ny, nx = flags.shape
    while (flags == SOLID).mean() < fraction:
        r = int(rng.integers(2, max(3, min(nx, ny, nz) // 6) + 1))
        c = [int(rng.integers(0, n)) for n in (nz, ny, nx)]
        lo = [max(0, c[k] - r) for k in range(3)]
        g = np.ogrid[tuple(slice(lo[k], min(flags.shape[k], c[k] + r + 1)) for k in range(3))]
        inside = sum((g[k] - c[k]) ** 2 for k in range(3)) < r * r
        flags[tuple(slice(lo[k], lo[k] + inside.shape[k]) for k in range(3))][inside] = SOLID
    return flags


@functools.lru_cache(maxsize=8)
def geometry(walls, nx, ny, nz, seed=0):
    """(flags, bc_values, periodic) of a box; flags (nz, ny, nx) uint8."""
    flags = np.zeros((nz, ny, nx), np.uint8)
    if walls == "periodic":
        return flags, None, (1, 1, 1)
    if walls == "cavity":  # moving lid on the top plane, outward normal +z
        flags[nz - 1] = VELOCITY | (4 << 3)
        return flags, np.tile(np.float32([0.05, 0, 0, 1]), (ny * nx, 1)), (0, 0, 0)
    if walls == "duct":  # solid spheres, periodic along x
        return _spheres(flags, 0.12, np.random.default_rng(seed)), None, (1, 0, 0)
    # "sphere": circular channel along x, sphere inside, inlet and outlet
    cy, cz, cx = ny // 2, nz // 2, nx // 4
    z, y, x = np.ogrid[:nz, :ny, :nx]
    radial = (y - cy) ** 2 + (z - cz) ** 2
    channel = np.broadcast_to(radial < (0.317 * ny) ** 2, flags.shape)
    flags[:] = OUTSIDE
    flags[channel] = FLUID
    flags[channel & (radial + (x - cx) ** 2 < (ny // 8) ** 2)] = SOLID
    flags[:, :, 0][channel[:, :, 0]] = VELOCITY | (1 << 3)      # normal -x
    flags[:, :, -1][channel[:, :, -1]] = PRESSURE | (0 << 3)    # normal +x
    bc = np.array([[0.04, 0, 0, 1] if f & 7 == VELOCITY else [0, 0, 0, 1]
                   for f in flags[flags & 6 == 2]], np.float32).reshape(-1, 4)
    return flags, bc, (0, 0, 0)


def level_map(nx, ny, nz):
    """Owning level per 32^3 cell: finest in the central quarter of z, level 1
    one eighth on either side, level 2 elsewhere."""
    z = (np.arange(nz // 32) * 32 + 16) / nz
    lv = np.where(abs(z - 0.5) < 0.125, 0, np.where(abs(z - 0.5) < 0.25, 1, 2)).astype(np.uint8)
    return np.ascontiguousarray(np.broadcast_to(lv[:, None, None], (nz // 32, ny // 32, nx // 32)))


def coarsen(rho, u):
    pool = functools.partial(torch.nn.functional.avg_pool3d, kernel_size=2)
    return pool(rho[None, None])[0, 0].contiguous(), pool(u[:, None])[:, 0].contiguous()


def network(seed, out_scale):
    """Flat FP32 parameters of the 16-64-64-1 network (W1, b1, W2, b2, W3, b3),
    He-initialised."""
    g = torch.Generator().manual_seed(seed + 1)
    z = functools.partial(torch.randn, generator=g, dtype=torch.float64)
    return torch.cat([z(1024) * math.sqrt(2 / 16), 0.1 * z(64), z(4096) * math.sqrt(2 / 64),
                      torch.zeros(64, dtype=torch.float64), z(64) * math.sqrt(1 / 64) * out_scale,
                      torch.zeros(1, dtype=torch.float64)])


def closure_network(seed):
    """A network for raw features: first-layer columns scaled by each
    feature's usual size, output of a few thousandths."""
    th = network(seed, 0.005)
    size = torch.tensor([1e-3, 3e-2, 3e-2, 3e-2] + [1e-2] * 8 + [1e-3] * 3 + [0.5], dtype=torch.float64)
    th[:1024] = (th[:1024].view(64, 16) / size).reshape(-1)
    return th.float()


@functools.lru_cache(maxsize=4)
def batch_members(n, lo, hi):
    """Mixed periodic grids: dims, flags, tau, kind per member."""
    rng = np.random.default_rng(7898)
    out = []
    for k in range(n):
        dims = tuple(int(8 * round(int(rng.integers(lo, hi + 1)) / 8)) for _ in range(3))
        frac, tau = float(rng.uniform(0, 0.2)), float(rng.uniform(0.52, 0.8))
        flags = _spheres(np.zeros(dims[::-1], np.uint8), frac, rng)
        out.append((dims, flags, tau, "dense" if k % 2 == 0 else "sparse"))
    return out


def _dims(case):
    return case["nx"], case["ny"], case["nz"]


def _physics(case, periodic, **more):
    return lbm.physics(case["tau"], case["collision"], case["storage"], periodic, lattice=case.get("q", 19), **more)


def _buffers(grid, storage):
    size = lbm.lbm_get_info(grid)["population_bytes"]
    return [torch.empty(b // BYTES[storage], dtype=DTYPE[storage], device=DEV) for b in size]


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("dense", "sparse"):
        dims = _dims(case)
        flags, bc, per = geometry("sphere" if kind == "sparse" else case["walls"], *dims)
        if kind == "dense":
            grid = lbm.lbm_grid_create_dense(dims, _physics(case, per))
            if case["walls"] != "periodic":
                lbm.lbm_set_boundary(grid, 0, flags, bc)
        else:
            grid = lbm.lbm_grid_create_sparse(dims, 8, flags, _physics(case, per))
            lbm.lbm_set_boundary(grid, 0, None, bc)
        lbm.lbm_init_equilibrium(grid, 0, *fields(dims, seed))
        return dict(case=case, grid=grid, out=_buffers(grid, case["storage"]))
    if kind == "multires":
        dims = _dims(case)
        grid = lbm.lbm_grid_create_multires(dims, 3, level_map(*dims), _physics(case, (1, 1, 1), closure=int(case["closure"])))
        if case["closure"]:
            lbm.lbm_closure_load(grid, closure_network(seed).numpy())
        rho, u = fields(dims, seed)
        for lv in range(3):
            lbm.lbm_init_equilibrium(grid, lv, rho, u)
            rho, u = coarsen(rho, u)
        return dict(case=case, grid=grid, out=_buffers(grid, case["storage"]))
    if kind == "batch":
        grids = []
        for k, (dims, flags, tau, how) in enumerate(batch_members(case["n"], case["lo"], case["hi"])):
            ph = lbm.physics(tau, case["collision"], case["storage"], (1, 1, 1))
            if how == "dense":
                g = lbm.lbm_grid_create_dense(dims, ph)
                lbm.lbm_set_boundary(g, 0, flags)
            else:
                g = lbm.lbm_grid_create_sparse(dims, 8, flags, ph)
            lbm.lbm_init_equilibrium(g, 0, *fields(dims, seed + k))
            grids.append(g)
        return dict(case=case, grids=grids, batch=lbm.lbm_batch_create(grids),
                    out=[_buffers(g, case["storage"])[0] for g in grids])
    if kind == "learn":
        dims = _dims(case)
        grid = lbm.lbm_grid_create_dense(dims, lbm.physics(case["tau"], storage=case["storage"], periodic=(1, 1, 1)))
        lbm.lbm_set_populations(grid, 0, checkpoint(dims, seed, case["tau"], case["storage"]))
        n = math.prod(dims) // case["r"] ** 3
        return dict(case=case, grid=grid, seed=seed, theta0=network(seed, 1.0).float().to(DEV),
                    theta=torch.empty(5313, dtype=torch.float32, device=DEV),
                    feats=torch.empty(n, 16, dtype=torch.float32, device=DEV),
                    targets=torch.empty(n, dtype=torch.float32, device=DEV))
    dims = _dims(case)
    grid = lbm.lbm_grid_create_dense(dims, lbm.physics(0.6, storage=case["storage"], periodic=(1, 1, 1), lattice=case["q"]))
    rho, u = fields(dims, seed)
    return dict(case=case, grid=grid, rho=rho, u=u, rho_out=torch.empty_like(rho), u_out=torch.empty_like(u))


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("dense", "sparse", "multires"):
        lbm.lbm_step(state["grid"], case["steps"])
        for lv, buf in enumerate(state["out"]):
            lbm.lbm_get_populations(state["grid"], lv, buf)
        return {"f%d" % lv: buf for lv, buf in enumerate(state["out"])}
    if kind == "batch":
        lbm.lbm_batch_step(state["batch"], case["steps"])
        for g, buf in zip(state["grids"], state["out"]):
            lbm.lbm_get_populations(g, 0, buf)
        return {"f%d" % k: buf for k, buf in enumerate(state["out"])}
    if kind == "learn":
        lbm.lbm_closure_dataset(state["grid"], case["r"], coarse_tau(case), state["feats"], state["targets"])
        state["theta"].copy_(state["theta0"])
        loss = lbm.lbm_closure_train(state["feats"], state["targets"], case["steps"], case["batch"], 1e-3,
                                     state["seed"], state["theta"])
        return {"feats": state["feats"], "targets": state["targets"], "theta": state["theta"],
                "loss": np.float32(loss)}
    lbm.lbm_init_equilibrium(state["grid"], 0, state["rho"], state["u"])
    lbm.lbm_get_moments(state["grid"], 0, state["rho_out"], state["u_out"])
    return {"rho": state["rho_out"], "u": state["u_out"], "sums": lbm.lbm_conservation(state["grid"])}


def coarse_tau(case):
    return 0.5 + (case["tau"] - 0.5) / case["r"]


def _updated(case):
    """(updated voxels of one pass, stored populations read out at its end)."""
    n = math.prod(_dims(case)) if "nx" in case else 0
    if case["kind"] == "dense":
        fl = geometry(case["walls"], *_dims(case))[0]
        return case["steps"] * int(((fl & 7) != SOLID).sum()), n
    if case["kind"] == "sparse":
        fl = geometry("sphere", *_dims(case))[0] & 7
        upd = (fl == FLUID) | (fl == VELOCITY) | (fl == PRESSURE)
        return case["steps"] * int(upd.sum()), len(_blocks(upd)[0]) * 512
    if case["kind"] == "multires":
        lm = level_map(*_dims(case))
        per = [int((lm == l).sum()) * 32 ** 3 // 8 ** l for l in range(3)]
        return case["steps"] * sum(p * 4 // 2 ** l for l, p in enumerate(per)), sum(per)
    members = batch_members(case["n"], case["lo"], case["hi"])
    return (case["steps"] * sum(int((fl != SOLID).sum()) for _, fl, _, _ in members),
            sum(math.prod(d) for d, _, _, _ in members))


def work(case):
    kind = case["kind"]
    if kind == "learn":
        n, nc = math.prod(_dims(case)), math.prod(_dims(case)) // case["r"] ** 3
        nets = 2 * (16 * 64 + 64 * 64 + 64)
        return {"bytes": 19 * BYTES[case["storage"]] * n + 2 * 17 * 4 * nc + case["steps"] * case["batch"] * 17 * 4,
                "flops": case["steps"] * case["batch"] * 3 * nets}
    if kind == "readout":
        n = math.prod(_dims(case))
        return {"bytes": 2 * n * 4 * 8 + 3 * n * case["q"] * BYTES[case["storage"]], "flops": 0}
    updates, slots = _updated(case)
    q, b = case.get("q", 19), BYTES[case["storage"]]
    return {"bytes": updates * 2 * q * b + 2 * slots * q * b, "flops": updates * 250 * q // 19}


# ----------------------------------------------------------- 64-bit evaluation

def _collide(g, tau, coll):
    """Post-collision populations of pulled g (Q, ...); tau a number or a field."""
    q, w = g.shape[0], weights(g.shape[0])
    rho = g.sum(0)
    u = torch.stack([sum(float(C[i][a]) * g[i] for i in range(q) if C[i][a]) for a in range(3)]) / rho
    eq = equilibrium(rho, u, q)
    om = 1.0 / tau
    if coll == "bgk":
        return g + om * (eq - g)
    return _regularize(eq, g - eq, om)


def _regularize(eq, d, om):
    q, w = d.shape[0], weights(d.shape[0])
    P = {(a, b): sum(float(C[i][a] * C[i][b]) * d[i] for i in range(q) if C[i][a] * C[i][b])
         for a in range(3) for b in range(a, 3)}
    tr = (P[0, 0] + P[1, 1] + P[2, 2]) / 3
    for i in range(q):
        s = sum((1 if a == b else 2) * float(C[i][a] * C[i][b]) * P[a, b] for a, b in P if C[i][a] * C[i][b])
        eq[i] += (1 - om) * 4.5 * w[i] * (s - tr)
    return eq


def _source_walls(flags, periodic, q):
    """(q, nz, ny, nx): the pull source of each population bounces back."""
    t = torch.from_numpy(flags & 7).to(DEV)
    wall = (t == SOLID) | (t == OUTSIDE)
    out = torch.zeros((q,) + flags.shape, dtype=torch.bool, device=DEV)
    for i in range(1, q):
        c = [int(v) for v in C[i]]
        out[i] = torch.roll(wall, (c[2], c[1], c[0]), (0, 1, 2))
        for a in range(3):
            if c[a] and not periodic[a]:
                edge = [slice(None)] * 3
                edge[2 - a] = 0 if c[a] > 0 else -1
                out[i][tuple(edge)] = True
    return out


def _pull(f, walls=None):
    g = torch.empty_like(f)
    for i in range(f.shape[0]):
        c = [int(v) for v in C[i]]
        g[i] = torch.roll(f[i], (c[2], c[1], c[0]), (0, 1, 2))
        if walls is not None and i:
            g[i] = torch.where(walls[i], f[opposite(i)], g[i])
    return g


def _boundary_nodes(g, out, flags, bc, om):
    """Regularized velocity / pressure nodes: out at their voxels from pulled g."""
    q = g.shape[0]
    where = np.flatnonzero(((flags & 7) == VELOCITY) | ((flags & 7) == PRESSURE))
    fl = flags.ravel()[where]
    vals = torch.from_numpy(bc.astype(np.float64)).to(DEV)
    for code in np.unique(fl):
        pick = torch.from_numpy(np.flatnonzero(fl == code)).to(DEV)
        idx = torch.from_numpy(where).to(DEV)[pick]
        axis, sign = (int(code) >> 3) // 2, 1 - 2 * ((int(code) >> 3) % 2)
        cn = [sign * int(C[i][axis]) for i in range(q)]
        s = g.view(q, -1)[:, idx].clone()
        total = sum(s[i] * (1 if cn[i] == 0 else 2) for i in range(q) if cn[i] >= 0)
        u = vals[pick, :3].T.clone()
        if code & 7 == VELOCITY:
            rho = total / (1 + sign * u[axis])
        else:
            rho = vals[pick, 3]
            u.zero_()
            u[axis] = sign * (total / rho - 1)
        eq = equilibrium(rho, u, q)
        for i in range(q):
            if cn[i] < 0:
                s[i] = eq[i] + s[opposite(i)] - eq[opposite(i)]
        out.view(q, -1)[:, idx] = _regularize(eq.clone(), s - eq, om)


def _evolve(f, flags, bc, periodic, tau, coll, steps):
    q = f.shape[0]
    plain = not (flags & 7).any()
    t = torch.from_numpy(flags & 7).to(DEV)
    still = (t == SOLID) | (t == OUTSIDE)
    walls = None if plain and all(periodic) else _source_walls(flags, periodic, q)
    f = torch.where(still, 0.0, f)
    for _ in range(steps):
        g = _pull(f, walls)
        f = _collide(g, tau, coll)
        if bc is not None:
            _boundary_nodes(g, f, flags, bc, 1.0 / tau)
        if not plain:
            f = torch.where(still, 0.0, f)
    return f, still


def _to_storage(f, still, storage):
    """Absolute populations as the buffers hold them; 0 where nothing is stored."""
    if storage != "f32":
        f = f - torch.tensor(weights(f.shape[0]), dtype=f.dtype, device=f.device).view(-1, 1, 1, 1)
    return torch.where(still, 0.0, f)


def _spread(v):
    v = v.astype(np.int64)
    return sum(((v >> b) & 1) << (3 * b) for b in range(10))


def _blocks(active, first=None):
    """(bz, by, bx) of the 8^3 blocks holding an active voxel, those marked
    `first` ahead, each group along the Morton curve."""
    pad = [(0, -n % 8) for n in active.shape]
    def any8(m):
        m = np.pad(m, pad)
        return m.reshape(m.shape[0] // 8, 8, m.shape[1] // 8, 8, m.shape[2] // 8, 8).any((1, 3, 5))
    has = any8(active)
    front = np.zeros_like(has) if first is None else (first if first.shape == has.shape else any8(first))
    z, y, x = np.nonzero(has)
    key = _spread(x) | (_spread(y) << 1) | (_spread(z) << 2) | (np.int64(~front[z, y, x]) << 40)
    order = np.argsort(key)
    return z[order], y[order], x[order]


def _to_blocks(f, blocks):
    q = f.shape[0]
    pad = [p for n in reversed(f.shape[1:]) for p in (0, -n % 8)]
    f = torch.nn.functional.pad(f, pad)
    nb = [n // 8 for n in f.shape[1:]]
    f = f.view(q, nb[0], 8, nb[1], 8, nb[2], 8).permute(1, 3, 5, 0, 2, 4, 6)
    z, y, x = (torch.from_numpy(v).to(DEV) for v in blocks)
    return f[z, y, x].reshape(-1)


def _features(g, tau):
    """The closure's 16 features per voxel of pulled populations, (16, ...)."""
    q = g.shape[0]
    rho = g.sum(0)
    u = torch.stack([sum(float(C[i][a]) * g[i] for i in range(q) if C[i][a]) for a in range(3)]) / rho
    d = g - equilibrium(rho, u, q)
    s = rho / 3
    P = {(a, b): sum(float(C[i][a] * C[i][b]) * d[i] for i in range(q) if C[i][a] * C[i][b]) / s
         for a in range(3) for b in range(a, 3)}
    third = [sum(float(C[i][a] * (C[i] ** 2).sum() - C[i][a] ** 3) * d[i] for i in range(7, q) if C[i][a]) / s
             for a in range(3)]
    tr = P[0, 0] + P[1, 1] + P[2, 2]
    norm = torch.sqrt(sum((1 if a == b else 2) * P[a, b] ** 2 for a, b in P))
    return torch.stack([rho - 1, u[0], u[1], u[2], P[0, 0], P[1, 1], P[2, 2], P[0, 1], P[0, 2], P[1, 2],
                        norm, tr] + third + [torch.full_like(rho, tau)])


def _layers(theta):
    return (theta[:1024].view(64, 16), theta[1024:1088], theta[1088:5184].view(64, 64), theta[5184:5248],
            theta[5248:5312], theta[5312])


def _exact_levels(case, seed):
    """Three levels, each on the virtual box of its own resolution.  Inside a
    step of level l, every voxel of it next to level l - 1 stands for 8
    virtual cells there, which stream for two finer steps without colliding."""
    dims = _dims(case)
    owner = np.kron(level_map(*dims), np.ones((4, 4, 4), np.uint8))  # per 8^3 finest block
    own, near, F, V = [], [], [], [None] * 3
    rho, u = fields(dims, seed)
    up = lambda a: a.repeat_interleave(2, -1).repeat_interleave(2, -2).repeat_interleave(2, -3)  # noqa: E731
    for lv in range(3):
        e = 2 ** lv
        m = np.kron(owner[::e, ::e, ::e] == lv, np.ones((8, 8, 8), bool))
        own.append(torch.from_numpy(m).to(DEV))
        finer = torch.from_numpy(np.kron(owner[::e, ::e, ::e] < lv, np.ones((8, 8, 8), bool))).to(DEV)
        for ax in range(3):
            finer = finer | torch.roll(finer, 1, ax) | torch.roll(finer, -1, ax)
        near.append(finer)
        F.append(torch.where(own[lv], absolute(stored(equilibrium(rho, u, 19), case["storage"]), 19), 0.0))
        rho, u = coarsen(rho, u)
    net = _layers(closure_network(seed).double().to(DEV)) if case["closure"] else None

    def advance(lv):
        tau = 0.5 + (case["tau"] - 0.5) / 2 ** lv
        state = F[lv] if V[lv] is None else F[lv] + V[lv]  # disjoint: own voxels, coarser neighbours' cells
        g = _pull(state)
        if V[lv] is not None:
            V[lv] = torch.where(over[lv], g, 0.0)
        if lv:
            V[lv - 1] = torch.where(over[lv - 1], up(F[lv]), 0.0)
            advance(lv - 1)
            advance(lv - 1)
            v = V[lv - 1]
            n = [k // 2 for k in v.shape[1:]]
            mean = v.view(19, n[0], 2, n[1], 2, n[2], 2).mean((2, 4, 6))
            g = torch.where(near[lv], mean, g)
        if net is not None and lv:
            cols = _features(g.view(19, -1)[:, own[lv].view(-1)], tau).T
            h = torch.relu(torch.relu(cols @ net[0].T + net[1]) @ net[2].T + net[3])
            field = torch.full(own[lv].shape, tau, dtype=torch.float64, device=DEV)
            field[own[lv]] = torch.clamp(tau + h @ net[4] + net[5], min=0.501)
            tau = field
        F[lv] = torch.where(own[lv], _collide(torch.where(own[lv], g, 1.0), tau, case["collision"]), 0.0)

    # cells of level lv's resolution that belong to level lv + 1
    over = [up(own[lv + 1]) if lv < 2 else None for lv in range(3)]
    for _ in range(case["steps"]):
        advance(2)
    out = {}
    for lv in range(3):
        e = 2 ** lv
        mine = owner[::e, ::e, ::e] == lv
        other = np.zeros_like(mine)
        for c in C[1:19]:
            other |= ~np.roll(mine, tuple(int(v) for v in c[::-1]), (0, 1, 2))
        blocks = _blocks(own[lv].cpu().numpy(), mine & other)
        out["f%d" % lv] = _to_blocks(_to_storage(F[lv], ~own[lv], case["storage"]), blocks)
    return out


def _box_mean(a, r):
    *lead, nz, ny, nx = a.shape
    return a.reshape(*lead, nz // r, r, ny // r, r, nx // r, r).mean((-5, -3, -1))


def _splitmix(x):
    x = x + np.uint64(0x9E3779B97F4A7C15)
    x = (x ^ (x >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    x = (x ^ (x >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return x ^ (x >> np.uint64(31))


def _exact_learn(case, seed):
    r, tau = case["r"], coarse_tau(case)
    f = absolute(checkpoint(_dims(case), seed, case["tau"], case["storage"]), 19)
    rho = f.sum(0)
    j = torch.stack([sum(float(C[i][a]) * f[i] for i in range(19) if C[i][a]) for a in range(3)])
    X = _features(_pull(_box_mean(f, r)), tau).reshape(16, -1).T.contiguous()
    rb, ub = _box_mean(rho, r), _box_mean(j, r) / _box_mean(rho, r)
    grad = [[0.5 * (torch.roll(ub[b], -1, 2 - a) - torch.roll(ub[b], 1, 2 - a)) for b in range(3)] for a in range(3)]
    t = [[_box_mean(j[a] * j[b] / rho, r) - rb * ub[a] * ub[b] for b in range(3)] for a in range(3)]
    tr = (t[0][0] + t[1][1] + t[2][2]) / 3
    num, den = torch.zeros_like(rb), torch.zeros_like(rb)
    for a in range(3):
        for b in range(3):
            S = 0.5 * (grad[a][b] + grad[b][a])
            num += (t[a][b] - (tr if a == b else 0)) * S
            den += 2 * rb * S * S
    for ax in range(3):
        num = num + torch.roll(num, 1, ax) + torch.roll(num, -1, ax)
        den = den + torch.roll(den, 1, ax) + torch.roll(den, -1, ax)
    T = torch.clamp(torch.where(den > 0, -3 * num / den, 0.0), -(tau - 0.5) + 1e-3, 0.5).reshape(-1)
    # standardise, train, fold
    n = T.numel()
    scale = lambda sd, mu: torch.where((sd > 1e-6 * mu.abs()) & (sd > 1e-30), sd, torch.ones_like(sd))  # noqa: E731
    mu, tm = X.mean(0), T.mean()
    sd, ts = scale(X.std(0, unbiased=False), mu), scale(T.std(unbiased=False), tm)
    Xs, Ts = (X - mu) / sd, (T - tm) / ts
    th = network(seed, 1.0).float().double().to(DEV)
    m, v = torch.zeros_like(th), torch.zeros_like(th)
    for k in range(1, case["steps"] + 1):
        with np.errstate(over="ignore"):
            at = _splitmix(np.arange(case["batch"], dtype=np.uint64) + np.uint64(seed + (k - 1) * case["batch"])) % np.uint64(n)
        idx = torch.from_numpy(at.astype(np.int64)).to(DEV)
        x, (W1, b1, W2, b2, W3, b3) = Xs[idx], _layers(th)
        z1 = x @ W1.T + b1
        h1 = torch.relu(z1)
        z2 = h1 @ W2.T + b2
        h2 = torch.relu(z2)
        res = h2 @ W3 + b3 - Ts[idx]
        loss = float((res * res).mean())
        dy = 2 * res / case["batch"]
        d2 = dy[:, None] * W3 * (z2 > 0)
        d1 = (d2 @ W2) * (z1 > 0)
        g = torch.cat([(d1.T @ x).reshape(-1), d1.sum(0), (d2.T @ h1).reshape(-1), d2.sum(0), h2.T @ dy, dy.sum()[None]])
        m = 0.9 * m + 0.1 * g
        v = 0.999 * v + 0.001 * g * g
        th = th - 1e-3 * (m / (1 - 0.9 ** k)) / (torch.sqrt(v / (1 - 0.999 ** k)) + 1e-8)
    W1, b1, W2, b2, W3, b3 = _layers(th)
    theta = torch.cat([(W1 / sd).reshape(-1), b1 - W1 @ (mu / sd), W2.reshape(-1), b2, W3 * ts, (b3 * ts + tm)[None]])
    return {"feats": X, "targets": T, "theta": theta, "loss": np.float64(loss)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "learn":
        return _exact_learn(case, seed)
    if kind == "multires":
        return _exact_levels(case, seed)
    if kind == "batch":
        out = {}
        for k, (dims, flags, tau, how) in enumerate(batch_members(case["n"], case["lo"], case["hi"])):
            f = absolute(stored(equilibrium(*fields(dims, seed + k), 19), case["storage"]), 19)
            f, still = _evolve(f, flags, None, (1, 1, 1), tau, case["collision"], case["steps"])
            # a batch stores the rest state in its solid voxels
            rest = f if case["storage"] != "f32" else torch.tensor(weights(19), dtype=f.dtype, device=DEV).view(-1, 1, 1, 1)
            f = _to_storage(f, still, case["storage"])
            if case["storage"] == "f32":
                f = torch.where(still, rest, f)
            out["f%d" % k] = f.reshape(-1) if how == "dense" else _to_blocks(f, _blocks(flags != SOLID))
        return out
    dims = _dims(case)
    rho, u = fields(dims, seed)
    if kind == "readout":
        f = absolute(stored(equilibrium(rho, u, case["q"]), case["storage"]), case["q"])
        m = f.sum(0)
        j = torch.stack([sum(float(C[i][a]) * f[i] for i in range(case["q"]) if C[i][a]) for a in range(3)])
        return {"rho": m, "u": j / m, "sums": torch.cat([m.sum()[None], j.sum((1, 2, 3))])}
    flags, bc, per = geometry("sphere" if kind == "sparse" else case["walls"], *dims)
    f = absolute(stored(equilibrium(rho, u, case["q"]), case["storage"]), case["q"])
    f, still = _evolve(f, flags, bc, per, case["tau"], case["collision"], case["steps"])
    f = _to_storage(f, still, case["storage"])
    if kind == "dense":
        return {"f0": f.reshape(-1)}
    t = flags & 7
    return {"f0": _to_blocks(f, _blocks((t == FLUID) | (t == VELOCITY) | (t == PRESSURE),
                                        (t == VELOCITY) | (t == PRESSURE)))}

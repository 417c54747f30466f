"""GPU: lbm_closure_dataset leaves no trace in the grid's buffers, whatever the
grid did before and does after, and its workspace comes from the grid's
allocator, goes back with the grid and may be refused."""
import numpy as np
import pytest

from paper_2503_07898_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
DIMS = (24, 16, 12)


def make(lbm, storage, allocator=None):
    rho, u = wl.turbulence(0, seed=6, u_rms=0.03, kmax=2, dims=DIMS)
    g = lbm.lbm_grid_create_dense(DIMS, lbm.physics(0.52, storage=storage, periodic=(1, 1, 1)), allocator)
    lbm.lbm_init_equilibrium(g, 0, rho, u)
    return g


def dataset(lbm, g, r):
    import torch
    n = int(np.prod(DIMS)) // r ** 3
    out = torch.empty(n, 16, device="cuda"), torch.empty(n, device="cuda")
    lbm.lbm_closure_dataset(g, r, 0.5 + 0.02 / r, *out)
    return out


def state(lbm, g):
    import torch
    t = torch.empty(lbm.lbm_get_info(g)["population_bytes"][0], dtype=torch.uint8, device="cuda")
    lbm.lbm_get_populations(g, 0, t)
    return t


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("before", [1, 2, 3])
@pytest.mark.parametrize("r", [1, 2, 4])
def test_walls_after_steps_and_a_dataset(lbm, storage, before, r):
    """The stored values of voxels that become solid are the older state's."""
    import torch
    flags = np.zeros(DIMS[::-1], np.uint8)
    flags[3:6, 4:9, 5:20] = 1
    a, b = make(lbm, storage), make(lbm, storage)
    for g in (a, b):
        lbm.lbm_step(g, before)
    dataset(lbm, a, r)
    for n in (1, 2):
        for g in (a, b):
            lbm.lbm_set_boundary(g, 0, flags, None)
            lbm.lbm_step(g, n)
        assert torch.equal(state(lbm, a), state(lbm, b))


def test_workspace_goes_through_the_allocator(lbm):
    import torch

    class Counting(lbm.TorchAllocator):
        live = 0
        limit = None

        def _alloc(self, ctx, nbytes, stream):
            if self.limit is not None and nbytes > self.limit:
                return None
            Counting.live += 1
            return super()._alloc(ctx, nbytes, stream)

        def _free(self, ctx, p, stream):
            Counting.live -= 1
            super()._free(ctx, p, stream)

    alloc = Counting()
    g = make(lbm, "f32", alloc)
    base = Counting.live
    want = dataset(lbm, g, 4)
    assert Counting.live == base + 1
    alloc.limit = 0                      # r = 2 needs more: refused, the call allocates for itself
    small = dataset(lbm, g, 2)
    alloc.limit = None
    for _ in range(2):
        assert all(torch.equal(x, y) for x, y in zip(dataset(lbm, g, 2), small))
    assert all(torch.equal(x, y) for x, y in zip(dataset(lbm, g, 4), want))
    assert Counting.live == base + 1
    lbm.lbm_grid_destroy(g)
    assert Counting.live == 0

"""The sweep preconditioner by lines and by items forms every value with the same operations in the same order: a mesh that
takes the first kernel, laid into a corner or the middle of one that is too large for it and zero elsewhere (no inflow from
there, as from the boundary), gives the same bits."""

import pytest

pytestmark = pytest.mark.gpu

LARGE = 77  # lines along the shorter side: one more than half of the 152 multiprocessors


@pytest.mark.parametrize("nx,nz,p,N,at", [(1, 1, 2, 4, (0, 0)), (9, 5, 2, 8, (3, 70)), (5, 9, 4, 16, (72, 0)), (12, 7, 6, 16, (30, 30)),
                                          (4, 6, 6, 16, (0, 71)), (5, 4, 8, 16, (72, 73))])
def test_lines_and_items_give_the_same_bits(lib, nx, nz, p, N, at):
    import torch
    ctx = lib.Context(p, N, 0.5, lib.ANG_FV0)
    g = torch.Generator(device="cuda")
    g.manual_seed(nx * 100 + nz)
    A = torch.randn(nz, nx, ctx.nin, ctx.nin, generator=g, device="cuda") * (0.5 / ctx.nin ** 0.5)
    r = torch.randn(nz, nx, ctx.nin, generator=g, device="cuda")
    z = torch.full_like(r, float("nan"))
    ctx.elrt_apply_precond(nx, nz, A, r, z)
    box = (slice(at[1], at[1] + nz), slice(at[0], at[0] + nx))
    big_A, big_r = torch.zeros(LARGE, LARGE, ctx.nin, ctx.nin, device="cuda"), torch.zeros(LARGE, LARGE, ctx.nin, device="cuda")
    big_A[box], big_r[box] = A, r
    big_z = torch.full_like(big_r, float("nan"))
    ctx.elrt_apply_precond(LARGE, LARGE, big_A, big_r, big_z)
    ctx.close()
    assert float(z.abs().max()) > 0 and torch.equal(big_z[box], z)
    big_z[box] = 0
    assert not bool(big_z.any())

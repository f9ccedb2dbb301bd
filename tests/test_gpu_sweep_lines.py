"""The sweep preconditioner's two kernels -- a mesh line per pair of CTAs, and items dealt round robin for meshes with
more lines than half the multiprocessors or elements too wide for two stages -- against the oracle, at the edges of
both: single elements, single lines along either axis, more lines than the first takes, one to four operator stages,
the widest elements, and a mesh on both sides of the square."""

import numpy as np
import pytest

from oracle import hdg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,nz,p,N", [(1, 1, 2, 4), (5, 1, 3, 8), (1, 6, 3, 8), (2, 17, 2, 12), (40, 3, 2, 4), (7, 7, 4, 16),
                                       (3, 2, 6, 16), (2, 3, 8, 16), (2, 2, 6, 28), (3, 2, 10, 32), (76, 77, 1, 4),
                                       (77, 78, 1, 4), (80, 2, 1, 4)])
def test_apply_matches_oracle(lib, nx, nz, p, N):
    import torch
    disc, mesh = hdg.Disc(p, N, 0.5, "fv0"), hdg.Mesh(nx, nz, 1.0)
    rng = np.random.default_rng(nx * 131 + nz)
    A32 = (rng.standard_normal((mesh.n_elems, disc.n_out, disc.n_in)) * (0.5 / np.sqrt(disc.n_in))).astype(np.float32)
    ctx = lib.Context(p, N, 0.5, 0)
    At = torch.tensor(A32, device="cuda")
    for k in range(3):  # repeated applications on other right-hand sides
        r = rng.standard_normal(mesh.n_elems * disc.n_out).astype(np.float32)
        z = torch.full((r.size,), float("nan"), dtype=torch.float32, device="cuda")
        ctx.elrt_apply_precond(nx, nz, At, torch.tensor(r, device="cuda"), z)
        ref = hdg.sweep_precond(mesh, disc, A32.astype(np.float64), r.astype(np.float64))
        # a value is a sum of n_in products, four sweeps deep: a few hundred FP32 roundings of the largest value
        np.testing.assert_allclose(z.cpu().numpy(), ref, rtol=0, atol=2e-5 * np.abs(ref).max())
    ctx.close()

"""The adjoint product itself (one-step TF32_IR builds with FP32 operators and nothing else asked for): both angular modes,
thick and thin elements and albedo 1, both product formats of the factorisation, chunked builds and any batch, one and two
operand stages, one to three column tiles."""

import numpy as np
import pytest

from oracle import hdg
from tests import _helpers as H

pytestmark = pytest.mark.gpu

HALF_ULP = 2.0 ** -24  # of a value's own power of two, at most this fraction of the value


def _build(lib, ctx, t, stats=False, refine=1):
    import torch
    n = t[1].numel()
    a = torch.full((n, ctx.nin, ctx.nin), float("nan"), device="cuda")
    m = torch.full((n, ctx.nm, ctx.nin), float("nan"), device="cuda")
    ctx.elrt_build_local(t[0], t[1], 1.0, a, m, mode=lib.LOCAL_TF32_IR, refine_steps=refine, h_elem=t[2], stats=stats)
    return a, m


def _beyond_rounding(x, ref):
    """Per element, the largest error that the rounding to FP32 does not explain."""
    e = np.abs(x.double().cpu().numpy() - ref)
    return np.maximum(e - HALF_ULP * np.abs(ref) * (1 + 1e-6), 0).max(axis=(1, 2))


@pytest.mark.parametrize("p,N,angular", [(2, 8, "do"), (4, 8, "fv0"), (4, 16, "do"), (6, 16, "fv0"), (6, 16, "do"), (8, 12, "fv0"),
                                         (8, 16, "do"), (6, 28, "fv0")])
def test_against_the_oracle_and_the_re_solve(lib, p, N, angular):
    """Either correction leaves a second-order error, the relative error of a second solution with the factors times the
    first solution's error: at most 1e-10 on the ordinary elements (the last four; the bar of a refined build).  Thick and
    thin ones leave more with a re-solve too.  The product's second solution is the first one, with FP16 operands in its
    backward sweep where the re-solve has TF32 ones, which costs a factor of about 10: up to 20 times the re-solve's error is
    allowed, far below the first solution's error (1e-6) or a lost column scale."""
    import torch
    k1, o1, h1 = H.thick_and_thin_elements(8, p, seed=500 + p)
    o1[2:5] = 1.0
    k2, o2, _ = H.random_elements(4, p, seed=p * N)
    kappa, omega, h = np.concatenate([k1, k2]), np.concatenate([o1, o2]), np.concatenate([h1, np.full(4, 0.2)])
    kappa = np.minimum(kappa, (400.0 / h)[:, None])  # entries within the range of the FP16 products
    d = hdg.Disc(p, N, 0.85, angular)
    ops = [d.local_operators(kappa[e] * h[e] / 2, float(omega[e])) for e in range(12)]
    ref = [np.stack([v[q] for v in ops]) for q in (0, 1)]
    ctx = lib.Context(p, N, 0.85, lib.ANG_FV0 if angular == "fv0" else lib.ANG_DO)
    t = [torch.tensor(v, device="cuda") for v in (kappa, omega, h)]
    for products in (lib.LU_PRODUCTS_AUTO, lib.LU_PRODUCTS_TF32):
        ctx.elrt_set_lu_products(products)
        ctx.elrt_profile_enable(True)
        ctx.elrt_profile_reset()
        adj = _build(lib, ctx, t)
        assert ctx.elrt_profile_get("adjoint")[1] == 1
        ctx.elrt_profile_enable(False)
        res = _build(lib, ctx, t, stats=True)
        for x, y, r in zip(adj, res, ref):
            ex, ey = _beyond_rounding(x, r), _beyond_rounding(y, r)
            assert (ex[8:] <= 1e-10).all(), (products, ex, ey)
            assert (ex <= 20 * ey + 1e-10).all(), (products, ex, ey)
    ctx.close()


@pytest.mark.parametrize("p,N", [(2, 8), (4, 16), (6, 16), (8, 12), (8, 16)])
def test_same_bits_in_any_batch_and_chunk(lib, p, N):
    import torch
    n = 330 if p < 8 else 160
    kappa, omega, h = H.random_elements(n, p, seed=3 * p + N)
    t = [torch.tensor(v, device="cuda") for v in (kappa, omega, np.full(n, h))]
    ctx = lib.Context(p, N, 0.85, lib.ANG_FV0)
    a, m = _build(lib, ctx, t)
    for part in (slice(0, 1), slice(100, 103), slice(n - 7, n)):
        b, r = _build(lib, ctx, [v[part].contiguous() for v in t])
        assert torch.equal(b, a[part]) and torch.equal(r, m[part])
    for chunk in (64, 7):
        ctx.elrt_set_tuning(chunk, 1, 12)
        b, r = _build(lib, ctx, t)
        assert torch.equal(b, a) and torch.equal(r, m)
    ctx.close()

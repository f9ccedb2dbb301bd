"""The refinement step of a build without statistics (FP32 operators: the adjoint product; FP64 operators: the
re-solve) against the FP64 oracle and against the same build with statistics: every element shape it takes, one and several column tiles, one and two
stages, both factorisations, both output types, both angular modes, and shapes beside them that keep the re-solve."""

import numpy as np
import pytest

from oracle import hdg
from tests import _helpers as H

pytestmark = pytest.mark.gpu

SHAPES = [(2, 8), (2, 12), (4, 8), (4, 12), (4, 16), (6, 8), (6, 12), (6, 16), (6, 28), (8, 8), (8, 12), (8, 16),
          (3, 8), (4, 20), (10, 32)]  # the last three: no kernel for the shape, or too wide for tensor memory


def _build(lib, ctx, t, mode, dtype, stats):
    import torch
    n = t[1].numel()
    a = torch.full((n, ctx.nin, ctx.nin), float("nan"), dtype=dtype, device="cuda")
    m = torch.full((n, ctx.nm, ctx.nin), float("nan"), dtype=dtype, device="cuda")
    ctx.elrt_build_local(t[0], t[1], 1.0, a, m, mode=mode, refine_steps=1, h_elem=t[2], stats=stats)
    return a.double().cpu().numpy(), m.double().cpu().numpy()


@pytest.mark.parametrize("mode", ["tf32", "fp32"])
@pytest.mark.parametrize("p,N", SHAPES)
def test_one_step_without_statistics(lib, p, N, mode):
    import torch
    if mode == "fp32" and (p, N) == (10, 32):
        pytest.skip("nu = 3872 is beyond the pivoted factorisation")
    mode = lib.LOCAL_TF32_IR if mode == "tf32" else lib.LOCAL_FP32_IR
    n = 1 if p == 10 else 5
    kappa, omega, _ = H.random_elements(n, p, seed=7 * p + N)
    h = np.full(n, 0.2)
    d = hdg.Disc(p, N, 0.85)
    ops = [d.local_operators(kappa[e] * h[e] / 2, float(omega[e])) for e in range(n)]
    o, q = np.stack([v[0] for v in ops]), np.stack([v[1] for v in ops])
    ctx = lib.Context(p, N, 0.85, lib.ANG_FV0)
    t = [torch.tensor(v, device="cuda") for v in (kappa, omega, h)]
    # ordinary elements: one step takes the FP32-level solution to the FP64 level, whichever way it is taken
    a, m = _build(lib, ctx, t, mode, torch.float64, False)
    np.testing.assert_allclose(a, o, atol=1e-10)
    np.testing.assert_allclose(m, q, atol=1e-10)
    a, m = _build(lib, ctx, t, mode, torch.float32, False)  # rounded once
    np.testing.assert_allclose(a, o, rtol=6.1e-8, atol=1e-10)
    np.testing.assert_allclose(m, q, rtol=6.1e-8, atol=1e-10)
    ctx.close()


@pytest.mark.parametrize("p,N", [(4, 8), (6, 16)])
def test_thick_and_thin_elements(lib, p, N):
    """The bounds of the one-step test with statistics, and the two ways against each other."""
    import torch
    kappa, omega, h = H.thick_and_thin_elements(14, p, seed=100 + p)
    omega[2:4] = 1.0
    d = hdg.Disc(p, N, 0.85)
    ops = [d.local_operators(kappa[e] * h[e] / 2, float(omega[e])) for e in range(14)]
    o, q = np.stack([v[0] for v in ops]), np.stack([v[1] for v in ops])
    ctx = lib.Context(p, N, 0.85, lib.ANG_FV0)
    t = [torch.tensor(v, device="cuda") for v in (kappa, omega, h)]
    for products in (lib.LU_PRODUCTS_AUTO, lib.LU_PRODUCTS_TF32):
        ctx.elrt_set_lu_products(products)
        a, m = _build(lib, ctx, t, lib.LOCAL_TF32_IR, torch.float32, False)
        np.testing.assert_allclose(a, o, atol=2e-6, rtol=2e-6)
        np.testing.assert_allclose(m, q, atol=2e-6, rtol=2e-6)
        a, m = _build(lib, ctx, t, lib.LOCAL_TF32_IR, torch.float64, False)
        b, r = _build(lib, ctx, t, lib.LOCAL_TF32_IR, torch.float64, True)
        for e in range(14):  # errors of the same size (the adjoint's solution is the same factorisation's)
            assert np.abs(a[e] - o[e]).max() <= 3 * np.abs(b[e] - o[e]).max() + 1e-11, e
            assert np.abs(m[e] - q[e]).max() <= 3 * np.abs(r[e] - q[e]).max() + 1e-11, e
    ctx.close()


def test_direction_samples_and_batches(lib):
    """Cell-centre directions; an element's operators do not depend on the batch it is in."""
    import torch
    p, N, n = 4, 16, 330
    kappa, omega, _ = H.random_elements(n, p, seed=5)
    d = hdg.Disc(p, N, 0.85, "do")
    ctx = lib.Context(p, N, 0.85, lib.ANG_DO)
    t = [torch.tensor(v, device="cuda") for v in (kappa, omega, np.full(n, 0.2))]
    a, m = _build(lib, ctx, t, lib.LOCAL_TF32_IR, torch.float64, False)
    for e in (0, 151, 152, 329):
        x = d.local_operators(kappa[e] * 0.1, float(omega[e]))
        np.testing.assert_allclose(a[e], x[0], atol=1e-10)
        np.testing.assert_allclose(m[e], x[1], atol=1e-10)
    few = [v[100:103].contiguous() for v in t]
    b, r = _build(lib, ctx, few, lib.LOCAL_TF32_IR, torch.float64, False)
    assert np.array_equal(b, a[100:103]) and np.array_equal(r, m[100:103])
    ctx.elrt_set_tuning(local_chunk=64)
    b, r = _build(lib, ctx, t, lib.LOCAL_TF32_IR, torch.float64, False)
    assert np.array_equal(b, a) and np.array_equal(r, m)
    ctx.close()

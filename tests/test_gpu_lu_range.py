"""The range in which the local factorisation forms its products in FP16: chunks whose largest assembled entry is above
it take 3xTF32 (the same bits as when the caller asks for that), chunks below it 3xFP16, and neither leaves FP16's range
on the elements whose factors and solutions grow most: thick, without absorption, isotropic, kappa inversely proportional
to the quadrature weights, everywhere or in a shell around a thin core."""

import numpy as np
import pytest

from oracle import hdg

pytestmark = pytest.mark.gpu


def _elements(d, largest):
    """kappa_hat of a thick element and of a thick shell whose largest assembled entry is `largest`, to within the transport
    part of a diagonal entry (below 1); albedo 1 and 0.999."""
    i = np.arange(d.nm)
    a, b = i % d.n1, i // d.n1
    edge = (a == 0) | (a == d.p) | (b == 0) | (b == d.p)
    m = (largest - 1.0) / max(1.0 - d.W[0, 0], d.W[0, 1])
    kh = np.stack([m / d.w2, m * np.where(edge, 1.0 / d.w2, 1e-9)])
    return np.repeat(kh, 2, axis=0), np.array([1.0, 0.999, 1.0, 0.999])


@pytest.mark.parametrize("p,N", [(4, 16), (6, 28), (8, 8), (8, 12), (8, 16)])
@pytest.mark.parametrize("refine,stats", [(0, False), (1, False), (1, True)])
def test_range_of_fp16_products(lib, p, N, refine, stats):
    import torch
    d = hdg.Disc(p, N, 0.0)
    ctx = lib.Context(p, N, 0.0, lib.ANG_FV0)
    for largest, f16 in ((1000.0, False), (500.0, False), (255.0, True)):
        kh, om = _elements(d, largest)
        k, o = torch.tensor(2.0 * kh, device="cuda"), torch.tensor(om, device="cuda")
        out = []
        for products in (lib.LU_PRODUCTS_AUTO, lib.LU_PRODUCTS_TF32):
            ctx.elrt_set_lu_products(products)
            a = torch.full((4, ctx.nin, ctx.nin), float("nan"), device="cuda")
            m = torch.full((4, ctx.nm, ctx.nin), float("nan"), device="cuda")
            ctx.elrt_build_local(k, o, 1.0, a, m, mode=lib.LOCAL_TF32_IR, refine_steps=refine, stats=stats)
            assert bool(torch.isfinite(a).all()) and bool(torch.isfinite(m).all()), (largest, products)
            out.append((a, m))
        same = torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
        assert same != f16, largest
    ctx.close()

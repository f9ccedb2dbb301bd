"""The float-float residual of every element shape with a kernel of its own, and of shapes beside them that take
the general kernel, against the FP64 oracle: thick, thin and ordinary elements, few (column chunks spread over
blocks) and one per block."""

import numpy as np
import pytest

from oracle import hdg
from tests import _helpers as H

pytestmark = pytest.mark.gpu

SHAPES = [(2, 8), (2, 12), (2, 16), (4, 8), (4, 12), (4, 16), (6, 8), (6, 12), (6, 16), (6, 28), (8, 8), (8, 12), (8, 16),
          (2, 4), (3, 8), (5, 12), (4, 20), (6, 24)]


@pytest.mark.parametrize("p,N", SHAPES)
def test_refined_operators_of_every_shape(lib, p, N):
    import torch
    k1, o1, h1 = H.thick_and_thin_elements(4, p, seed=300 + p)
    k2, o2, _ = H.random_elements(2, p, seed=p + N)
    kappa, omega, h = np.concatenate([k1, k2]), np.concatenate([o1, o2]), np.concatenate([h1, np.full(2, 0.2)])
    d = hdg.Disc(p, N, 0.85)
    ops = [d.local_operators(kappa[e] * h[e] / 2, float(omega[e])) for e in range(6)]
    for copies in (1, 52):  # 6 elements, and more elements than two blocks per multiprocessor hold
        n = 6 * copies
        ctx = lib.Context(p, N, 0.85, lib.ANG_FV0)
        a = torch.empty(n, ctx.nin, ctx.nin, dtype=torch.float64, device="cuda")
        m = torch.empty(n, ctx.nm, ctx.nin, dtype=torch.float64, device="cuda")
        t = [torch.tensor(np.concatenate([v] * copies), device="cuda") for v in (kappa, omega, h)]
        st = ctx.elrt_build_local(t[0], t[1], 1.0, a, m, mode=lib.LOCAL_TF32_IR, refine_steps=2, h_elem=t[2])
        ctx.close()
        assert st.n_flagged == 0 and st.max_rel_residual < 1e-12, st.max_rel_residual
        for e in range(6):
            np.testing.assert_allclose(a[e::6].cpu().numpy(), np.broadcast_to(ops[e][0], (copies, *ops[e][0].shape)), atol=1e-10)
            np.testing.assert_allclose(m[e::6].cpu().numpy(), np.broadcast_to(ops[e][1], (copies, *ops[e][1].shape)), atol=1e-10)


@pytest.mark.parametrize("p,N", [(2, 8), (4, 12), (6, 16), (8, 16)])
@pytest.mark.parametrize("steps", [1, 2])
def test_residual_does_not_depend_on_the_batch(lib, p, N, steps):
    """However many blocks share an element's columns (a rule on the batch size), the arithmetic of a column is the
    same: copies of one element come out with the bits of the element alone."""
    import torch
    k, o, _ = H.random_elements(1, p, seed=40 + p)
    ctx = lib.Context(p, N, 0.85, lib.ANG_FV0)
    first = None
    for n in (1, 7, 77, 153, 305, 481):
        a = torch.empty(n, ctx.nin, ctx.nin, dtype=torch.float64, device="cuda")
        m = torch.empty(n, ctx.nm, ctx.nin, dtype=torch.float64, device="cuda")
        kappa, omega = torch.tensor(np.repeat(k, n, 0), device="cuda"), torch.tensor(np.repeat(o, n), device="cuda")
        st = ctx.elrt_build_local(kappa, omega, 0.3, a, m, mode=lib.LOCAL_TF32_IR, refine_steps=steps)
        if first is None:
            first = a[0].clone(), m[0].clone(), st.max_rel_residual
        assert torch.equal(a, first[0].expand_as(a)) and torch.equal(m, first[1].expand_as(m))
        assert st.max_rel_residual == first[2]
    ctx.close()

"""The pivoted LU takes 256 or 512 threads per element, by the size of the system and of the batch: the operators of an
element have the same bits either way, on both sides of the sizes where two panels fit a multiprocessor."""

import numpy as np
import pytest

from tests import _helpers as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,N,dtype", [(3, 20, "fp32"), (4, 16, "fp32"), (6, 12, "fp32"), (8, 8, "fp32"), (3, 20, "fp64"), (6, 8, "fp64"),
                                       (6, 16, "fp64")])
def test_same_bits_in_small_and_large_batches(lib, p, N, dtype):
    import torch
    kappa, omega, h = H.random_elements(3, p, seed=p + N)
    ctx = lib.Context(p, N, 0.85, lib.ANG_FV0)
    out = []
    for copies in (1, 54):  # 3 elements, and more than one per multiprocessor
        a = torch.empty(3 * copies, ctx.nin, ctx.nin, dtype=torch.float64, device="cuda")
        m = torch.empty(3 * copies, ctx.nm, ctx.nin, dtype=torch.float64, device="cuda")
        ctx.elrt_build_local(torch.tensor(np.tile(kappa, (copies, 1)), device="cuda"), torch.tensor(np.tile(omega, copies), device="cuda"),
                             h, a, m, mode=lib.LOCAL_FP64 if dtype == "fp64" else lib.LOCAL_FP32_IR, refine_steps=1)
        out.append((a.reshape(copies, 3, -1), m.reshape(copies, 3, -1)))
    ctx.close()
    for few, many in zip(*out):
        assert torch.equal(many, few.expand_as(many))

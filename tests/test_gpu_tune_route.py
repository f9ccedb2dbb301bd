"""The autotuner times the build that the pipeline runs: with one refinement step, elrt_solve_field (as the binding calls it)
and elrt_solve_batch re-solve, so no candidate takes the adjoint product instead."""

import pytest

from tests import _helpers as H

pytestmark = pytest.mark.gpu


def test_autotune_times_the_pipelines_build(lib):
    import torch
    prob = H.small_cloud(5, 4, 6, 16)
    kap, om, g = (torch.tensor(v, device="cuda") for v in (H.lib_kappa(prob), prob.omega, prob.inflow))
    ctx = lib.Context(prob.p, prob.n_angles, prob.hg_g, lib.ANG_FV0)
    counts = []
    for call in ("field", "tune"):
        ctx.elrt_profile_enable(True)
        ctx.elrt_profile_reset()
        if call == "field":
            mean = torch.empty(prob.nx * prob.nz, ctx.nm, dtype=torch.float64, device="cuda")
            ctx.elrt_solve_field(prob.nx, prob.nz, prob.h, kap, om, g, mean, mode=lib.LOCAL_TF32_IR, refine_steps=1, rtol=1e-8)
        else:
            ctx.elrt_autotune(prob.nx, prob.nz, prob.h, kap, om, g, mode=lib.LOCAL_TF32_IR, refine_steps=1, rtol=1e-8)
        # residuals per build: two with a re-solve, one with the adjoint product
        counts.append([ctx.elrt_profile_get(k)[1] for k in ("assemble", "residual", "adjoint")])
    ctx.close()
    (builds, res, adj), (t_builds, t_res, t_adj) = counts
    assert t_builds == 7 and res == 2 * builds and t_res == 2 * t_builds and adj == t_adj == 0

"""Which builds take their refinement step as an adjoint product: TF32_IR with one step and FP32 operators, when the caller
asks for nothing else.  Every other build re-solves, FP32_IR with CUDA-core arithmetic throughout."""

import pytest

from tests import _helpers as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode,steps,dtype,extra,adjoint", [
    ("tf32", 1, "float32", None, True), ("tf32", 1, "float32", "stats", False), ("tf32", 1, "float32", "status", False),
    ("tf32", 1, "float32", "rad", False), ("tf32", 1, "float64", None, False), ("tf32", 2, "float32", None, False),
    ("tf32", 0, "float32", None, False), ("fp32", 1, "float32", None, False), ("fp32", 1, "float32", "stats", False),
    ("fp32", 2, "float32", None, False)])
def test_route(lib, mode, steps, dtype, extra, adjoint):
    import torch
    p, N, n = 6, 16, 3
    kappa, omega, h = H.random_elements(n, p, seed=11)
    ctx = lib.Context(p, N, 0.85, lib.ANG_FV0)
    dt = getattr(torch, dtype)
    a, m = torch.empty(n, ctx.nin, ctx.nin, device="cuda", dtype=dt), torch.empty(n, ctx.nm, ctx.nin, device="cuda", dtype=dt)
    ctx.elrt_profile_enable(True)
    kw = {"in2rad": torch.empty(n, ctx.nu, ctx.nin, device="cuda", dtype=dt)} if extra == "rad" else {}
    build = ctx.elrt_build_local_ex if extra == "rad" else ctx.elrt_build_local
    build(torch.tensor(kappa, device="cuda"), torch.tensor(omega, device="cuda"), h, a, m,
          mode=lib.LOCAL_TF32_IR if mode == "tf32" else lib.LOCAL_FP32_IR, refine_steps=steps, stats=extra == "stats",
          elem_status=torch.empty(n, dtype=torch.int32, device="cuda") if extra == "status" else None, **kw)
    launches = {k: ctx.elrt_profile_get(k)[1] for k in ("adjoint", "lu_factor_solve", "lu_resolve", "lu_tc_update")}
    ctx.close()
    assert launches["adjoint"] == (1 if adjoint else 0)
    if mode == "fp32":  # no tensor-core kernel at all
        assert launches["lu_factor_solve"] == 1 and launches["lu_resolve"] == steps and launches["lu_tc_update"] == 0
    else:
        assert launches["lu_factor_solve"] == launches["lu_resolve"] == 0 and launches["lu_tc_update"] > 0

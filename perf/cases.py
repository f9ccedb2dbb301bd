"""What the performance of the library is measured on: calls of its public entry points as its users make them.

A case is a dict of plain values; `kind` says which call it is:

  build      elrt_build_local: in2out / in2sol of a batch of elements (TF32_IR or FP32_IR)
  emission   elrt_build_local_ex: the same with a volume source and the radiance operator A_i2u
  unit       the plain FP64 path on a small mesh: elrt_build_local, elrt_solve_global, elrt_recover_mean
  skeleton   elrt_solve_global and elrt_recover_mean on operators that are in hand
  batch      elrt_solve_batch: Algorithm 1 on several uneven fields of several degrees in one call
  infer      elrt_net_infer: learned in2out / in2sol of a batch of elements
  train      elrt_net_train_step (forward, backward, Adam), then the updated network's outputs

Sizes come from the repository's workloads and benchmark (the 64 x 64 Gaussian-cloud slab at p = 6 with
16 angles, uneven fields with p in {4, 6, 8}, random elements for the network, the 4 x 1024 network, the
Legendre-modal training recipe with 28 angles and width 128, the 4 x 4 unit square).
"""

import math

import numpy as np
import torch

import paper_2308_02467_gb300 as E

DEV = "cuda"
MODES = {"tf32": E.LOCAL_TF32_IR, "fp32": E.LOCAL_FP32_IR}


def listed():
    return [
        # the plain FP64 classical method on a tiny mesh: the smallest call, bound by latency and launches
        {"name": "unit_square_fp64", "kind": "unit", "nx": 4, "nz": 4, "p": 4, "N": 8},
        # the classical fallback of a learned field: a handful of elements, one refinement sweep
        {"name": "build_fallback_9", "kind": "build", "field": "random", "mode": "tf32", "E": 9, "p": 6, "N": 16,
         "refine": 1, "stats": False},
        # the benchmark slab's local stage: 64 x 64 elements, one refinement sweep
        {"name": "build_slab_64x64", "kind": "build", "field": "slab", "mode": "tf32", "E": 4096, "p": 6, "N": 16,
         "refine": 1, "stats": False},
        # a field of the uneven batch at its highest degree, with the statistics a careful caller asks for
        {"name": "build_uneven_p8", "kind": "build", "field": "slab", "mode": "tf32", "E": 29 * 43, "p": 8, "N": 16,
         "refine": 1, "stats": True},
        # training labels for the network: random elements, FP32 LU with pivoting, the binding's defaults otherwise
        {"name": "labels_fp32", "kind": "build", "field": "random", "mode": "fp32", "E": 777, "p": 6, "N": 16,
         "refine": 1, "stats": True},
        # thermal emission: volume source, radiance operator
        {"name": "emission_radiance", "kind": "emission", "E": 24 * 20, "p": 6, "N": 16, "refine": 1},
        # the benchmark slab's skeleton solve with the entry point's own tolerance, and the recovery
        {"name": "skeleton_64x64", "kind": "skeleton", "nx": 64, "nz": 64, "p": 6, "N": 16},
        # an elongated field of odd sides
        {"name": "skeleton_127x17_p4", "kind": "skeleton", "nx": 127, "nz": 17, "p": 4, "N": 16},
        # several uneven fields in one call
        {"name": "batch_uneven", "kind": "batch", "nx4": 37, "nz4": 52, "nx6": 24, "nz6": 41, "nx8": 16, "nz8": 23, "N": 16},
        # the learned local stage of the benchmark slab
        {"name": "infer_4096", "kind": "infer", "E": 4096, "p": 6, "N": 16, "width": 1024, "hidden": 4, "act": "gelu"},
        # one training step of that network at its batch size
        {"name": "train_1024", "kind": "train", "B": 1024, "p": 6, "N": 16, "width": 1024, "hidden": 4, "act": "gelu"},
        # one training step of the Legendre-modal recipe: 28 angles, width 128, batch 64
        {"name": "train_modal_64", "kind": "train", "B": 64, "p": 6, "N": 28, "width": 128, "hidden": 3, "act": "elu"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["build", "build", "build", "emission", "unit", "skeleton", "batch", "infer", "train"])
    if kind == "build":
        mode = rng.choice(["tf32", "tf32", "fp32"])
        p = rng.choice([2, 4, 6, 8])
        N = rng.choice([8, 12, 16]) if p == 8 else rng.choice([8, 12, 16, 28])
        nu = (p + 1) ** 2 * N
        most = max(8, min(4096, int((1.5e12 if mode == "tf32" else 4e11) / nu ** 3)))
        return {"kind": kind, "field": rng.choice(["slab", "random"]), "mode": mode, "E": _log_int(rng, 1, most), "p": p,
                "N": N, "refine": rng.choice([1, 1, 2]), "stats": rng.random() < 0.4}
    if kind == "emission":
        p = rng.choice([2, 4, 6])
        return {"kind": kind, "E": _log_int(rng, 4, 600), "p": p, "N": rng.choice([8, 16]), "refine": rng.choice([1, 2])}
    if kind == "unit":
        return {"kind": kind, "nx": rng.randint(1, 8), "nz": rng.randint(1, 8), "p": rng.choice([2, 3, 4]), "N": rng.choice([4, 8])}
    if kind == "skeleton":
        return {"kind": kind, "nx": _log_int(rng, 3, 64), "nz": _log_int(rng, 3, 64), "p": rng.choice([2, 4, 6]),
                "N": rng.choice([8, 12, 16])}
    if kind == "batch":
        return {"kind": kind, "nx4": rng.randint(16, 40), "nz4": rng.randint(16, 40), "nx6": rng.randint(16, 32),
                "nz6": rng.randint(16, 32), "nx8": rng.randint(4, 18), "nz8": rng.randint(4, 18), "N": rng.choice([8, 16])}
    if kind == "infer":
        return {"kind": kind, "E": _log_int(rng, 1, 4096), "p": rng.choice([4, 6]), "N": 16, "width": rng.choice([128, 256, 1024]),
                "hidden": rng.randint(1, 4), "act": rng.choice(["gelu", "elu"])}
    return {"kind": kind, "B": 64 * rng.choice([1, 2, 3, 5, 8, 16]), "p": rng.choice([4, 6]), "N": rng.choice([8, 16]),
            "width": rng.choice([128, 256, 1024]), "hidden": rng.randint(1, 4), "act": rng.choice(["gelu", "elu"])}


# ---------------------------------------------------------------------------------------------- inputs

def _gen(seed, salt=0):
    g = torch.Generator(device=DEV)
    g.manual_seed(1_000_003 * (int(seed) % 2_000_003) + salt)
    return g


def _uni(g, lo, hi, *shape):
    return lo + (hi - lo) * torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64)


def _lgl(p):
    """LGL nodes and weights, and D[m, a] = l_a'(x_m), from numpy's Legendre module."""
    leg = np.polynomial.legendre
    c = np.zeros(p + 1)
    c[p] = 1.0
    x = np.concatenate([[-1.0], np.sort(np.real(leg.legroots(leg.legder(c)))), [1.0]])
    for _ in range(4):
        x[1:-1] -= leg.legval(x[1:-1], leg.legder(c)) / leg.legval(x[1:-1], leg.legder(c, 2))
    w = 2.0 / (p * (p + 1) * leg.legval(x, c) ** 2)
    V = leg.legvander(x, p)
    dV = np.stack([leg.legval(x, leg.legder(np.eye(p + 1)[j])) if j else np.zeros(p + 1) for j in range(p + 1)], axis=1)
    return x, w, dV @ np.linalg.inv(V)


def _slab_kappa(g, nx, nz, p, first=0, count=None):
    """1 to 5 Gaussian clouds on a background of 0.1 in a slab of 10 km, at the nodes of elements first .. first + count."""
    x = torch.tensor(_lgl(p)[0], device=DEV)
    h = 10.0 / max(nx, nz)
    n = 1 + int(torch.randint(0, 5, (1,), generator=g, device=DEV))
    amp, wid = _uni(g, 1.0, 30.0, n), _uni(g, 0.5, 3.0, n)
    cx, cz = _uni(g, 0.0, nx * h, n), _uni(g, 0.0, nz * h, n)
    e = torch.arange(first, first + (nx * nz if count is None else count), device=DEV)
    X = (((e % nx).double()[:, None, None] + 0.5 * (x[None, None, :] + 1.0)) * h).expand(-1, p + 1, -1)
    Z = ((torch.div(e, nx, rounding_mode="floor").double()[:, None, None] + 0.5 * (x[None, :, None] + 1.0)) * h).expand(-1, -1, p + 1)
    k = torch.full_like(X, 0.1)
    for j in range(n):
        k = k + amp[j] * torch.exp(-((X - cx[j]) ** 2 + (Z - cz[j]) ** 2) / (2.0 * wid[j] ** 2))
    return k.reshape(e.numel(), -1).contiguous(), h


def _random_elements(g, n, p, modes=16):
    """Independent elements: side U[0.05, 1] km, lognormal kappa from random Fourier features, albedo U[0.9, 1]."""
    x = torch.tensor(_lgl(p)[0], device=DEV)
    h, mu, sd = _uni(g, 0.05, 1.0, n), _uni(g, -2.0, 3.5, n), _uni(g, 0.0, 1.5, n)
    ell = _uni(g, 0.1, 2.0, n) * h
    kv = torch.randn(n, modes, 2, generator=g, device=DEV, dtype=torch.float64) / ell[:, None, None]
    ph = _uni(g, 0.0, 2.0 * math.pi, n, modes)
    xx = (0.5 * h)[:, None] * x[None, :]
    arg = (kv[:, :, 0, None, None] * xx[:, None, None, :] + kv[:, :, 1, None, None] * xx[:, None, :, None]
           + ph[:, :, None, None])
    f = torch.cos(arg).sum(dim=1) * math.sqrt(2.0 / modes)
    kappa = torch.exp(mu[:, None, None] + sd[:, None, None] * f).reshape(n, -1).contiguous()
    return kappa, _uni(g, 0.9, 1.0, n), h


def _beam(nx, nz, p, N, theta=300.0):
    """Collimated beam entering through the top: one angular cell carries N / (2 pi)."""
    half, q = N // 2, N // 4
    g = torch.zeros(2 * (nx + nz), p + 1, half, device=DEV, dtype=torch.float64)
    g[nx + nz:2 * nx + nz, :, int(theta * N / 360.0 + 1e-9) - 2 * q] = N / (2.0 * math.pi)
    return g.reshape(-1).contiguous()


def _inputs(case, seed):
    """The physical inputs of a case, from the seed alone."""
    g, k = _gen(seed), case["kind"]
    if k == "build":
        n, p = case["E"], case["p"]
        if case["field"] == "random":
            kappa, omega, h = _random_elements(g, n, p)
            return {"kappa": kappa, "omega": omega, "h": 1.0, "h_elem": h}
        nx = max(1, int(math.sqrt(n)))
        nz = -(-n // nx)
        kappa, h = _slab_kappa(g, nx, nz, p, 0, n)
        return {"kappa": kappa, "omega": torch.full((n,), 0.99, device=DEV, dtype=torch.float64), "h": h, "h_elem": None}
    if k == "emission":
        n, p, N = case["E"], case["p"], case["N"]
        nx = max(1, int(math.sqrt(n)))
        nz = -(-n // nx)
        kappa, h = _slab_kappa(g, nx, nz, p, 0, n)
        omega = _uni(g, 0.9, 1.0, n)
        height = torch.div(torch.arange(n, device=DEV), nx, rounding_mode="floor").double() / nz
        f = ((1.0 - omega) * (1.0 + height))[:, None, None] * kappa[:, None, :]
        return {"kappa": kappa, "omega": omega, "h": h, "source": f.expand(-1, N, -1).contiguous()}
    if k == "unit":
        n = case["nx"] * case["nz"]
        kappa = torch.full((n, (case["p"] + 1) ** 2), 1.0, device=DEV, dtype=torch.float64) * _uni(g, 0.5, 2.0, 1)
        return {"kappa": kappa, "omega": torch.zeros(n, device=DEV, dtype=torch.float64), "h": 1.0 / max(case["nx"], case["nz"]),
                "g": _beam(case["nx"], case["nz"], case["p"], case["N"])}
    if k == "skeleton":
        kappa, h = _slab_kappa(g, case["nx"], case["nz"], case["p"])
        return {"kappa": kappa, "omega": torch.full((case["nx"] * case["nz"],), 0.99, device=DEV, dtype=torch.float64), "h": h,
                "g": _beam(case["nx"], case["nz"], case["p"], case["N"])}
    if k == "batch":
        fields = []
        for p in (4, 6, 8):
            nx, nz = case["nx%d" % p], case["nz%d" % p]
            kappa, h = _slab_kappa(g, nx, nz, p)
            omega = torch.ones(nx * nz, device=DEV, dtype=torch.float64) * _uni(g, 0.9, 0.995, 1)
            fields.append((nx, nz, h, kappa, omega, _beam(nx, nz, p, case["N"])))
        return {"fields": fields}
    p, N = case["p"], case["N"]
    nm, nin = (p + 1) ** 2, 2 * (p + 1) * N
    nout, nf = nin * nin + nm * nin, nm + 1
    fpad = (nf + 63) // 64 * 64
    weights, nl = [], case["hidden"] + 1
    for l in range(nl):
        out, inp, pad = (nout if l == nl - 1 else case["width"]), (nf if l == 0 else case["width"]), (fpad if l == 0 else case["width"])
        b = 1.0 / math.sqrt(inp)
        W = (torch.rand(out, pad, generator=g, device=DEV) * 2.0 - 1.0) * b
        W[:, inp:] = 0.0
        weights.append((W, (torch.rand(out, generator=g, device=DEV) * 2.0 - 1.0) * b))
    if k == "infer":
        kappa, omega, h = _random_elements(g, case["E"], p)
        fit = _random_elements(g, 64, p)
        labels = (torch.randn(64, nin * nin, generator=g, device=DEV) * 0.1, torch.randn(64, nm * nin, generator=g, device=DEV) * 0.1)
        return {"weights": weights, "kappa": kappa, "omega": omega, "h": h, "fit": fit, "labels": labels}
    x = torch.zeros(case["B"], fpad, device=DEV)
    x[:, :nf] = torch.randn(case["B"], nf, generator=g, device=DEV)
    return {"weights": weights, "x": x, "t": torch.randn(case["B"], nout, generator=g, device=DEV)}


# ---------------------------------------------------------------------------------------------- prepare, run

def _net(case, weights):
    net = E.Net(case["p"], case["N"], n_hidden=case["hidden"], width=case["width"], activation=case["act"], seed=1)
    return net


def _set_weights(net, weights):
    for l, (W, b) in enumerate(weights):
        net.elrt_net_params(l, "W", W.cpu().numpy())
        net.elrt_net_params(l, "b", b.cpu().numpy())


def _f64(*shape):
    return torch.empty(*shape, device=DEV, dtype=torch.float64)


def prepare(case, seed):
    d, k = _inputs(case, seed), case["kind"]
    s = {"case": case, **{q: v for q, v in d.items() if q not in ("weights", "fit", "labels")}}
    if k == "batch":
        s["ctxs"] = [E.Context(p, case["N"], 0.85) for p in (4, 6, 8)]
        s["means"] = [_f64(f[0] * f[1], c.nm) for f, c in zip(s["fields"], s["ctxs"])]
        return s
    if k in ("infer", "train"):
        net = s["net"] = _net(case, d["weights"])
        if k == "infer":
            kf, of, hf = d["fit"]
            net.elrt_net_fit(kf, of, hf, d["labels"][0], d["labels"][1], epochs=1, batch=64, lr=1e-30)  # the standardisation
            s["i2o"] = torch.empty(case["E"], net.nin, net.nin, device=DEV)
            s["i2m"] = torch.empty(case["E"], net.nm, net.nin, device=DEV)
        else:
            s["y"] = torch.empty(case["B"], net.n_out, device=DEV)
        _set_weights(net, d["weights"])
        return s
    p, N = case["p"], case["N"]
    n = case["E"] if "E" in case else case["nx"] * case["nz"]
    ctx = s["ctx"] = E.Context(p, N, 0.0 if k == "unit" else 0.85)
    dt = torch.float64 if k == "unit" else torch.float32
    s["i2o"] = torch.empty(n, ctx.nin, ctx.nin, device=DEV, dtype=dt)
    s["i2m"] = torch.empty(n, ctx.nm, ctx.nin, device=DEV, dtype=dt)
    if k == "emission":
        s["f2o"], s["f2m"], s["f2u"] = _f64(n, ctx.nin), _f64(n, ctx.nm), _f64(n, ctx.nu)
        s["rad"] = torch.empty(n, ctx.nu, ctx.nin, device=DEV)
    if k in ("unit", "skeleton"):
        s["sk"], s["mean"] = _f64(n, ctx.nin), _f64(n, ctx.nm)
    if k == "skeleton":  # the operators in hand: refined until only their rounding to FP32 is left
        c = E.Context(p, N, 0.85)
        c.elrt_build_local(s["kappa"], s["omega"], s["h"], s["i2o"], s["i2m"], mode=E.LOCAL_TF32_IR, refine_steps=3)
        c.close()
    return s


def run(s):
    case, k = s["case"], s["case"]["kind"]
    if k == "build":
        s["ctx"].elrt_build_local(s["kappa"], s["omega"], s["h"], s["i2o"], s["i2m"], mode=MODES[case["mode"]],
                                  refine_steps=case["refine"], h_elem=s["h_elem"], stats=case["stats"])
        return s["i2o"], s["i2m"]
    if k == "emission":
        s["ctx"].elrt_build_local_ex(s["kappa"], s["omega"], s["h"], s["i2o"], s["i2m"], mode=E.LOCAL_TF32_IR,
                                     refine_steps=case["refine"], source=s["source"], f2o=s["f2o"], f2m=s["f2m"], f2u=s["f2u"],
                                     in2rad=s["rad"], stats=False)
        return s["i2o"], s["i2m"], s["f2o"], s["f2m"], s["f2u"], s["rad"]
    if k in ("unit", "skeleton"):
        c = s["ctx"]
        if k == "unit":
            c.elrt_build_local(s["kappa"], s["omega"], s["h"], s["i2o"], s["i2m"], mode=E.LOCAL_FP64)
        c.elrt_solve_global(case["nx"], case["nz"], s["i2o"], s["g"], s["sk"])
        c.elrt_recover_mean(case["nx"], case["nz"], s["i2m"], s["sk"], s["g"], s["mean"])
        return s["sk"], s["mean"]
    if k == "batch":
        E.elrt_solve_batch(s["ctxs"], s["fields"], [0, 1, 2], s["means"], mode=E.LOCAL_TF32_IR, refine_steps=2, rtol=1e-10)
        return s["means"]
    if k == "infer":
        s["net"].elrt_net_infer(s["kappa"], s["omega"], 1.0, s["i2o"], s["i2m"], h_elem=s["h"])
        return s["i2o"], s["i2m"]
    net = s["net"]
    loss = net.elrt_net_train_step(s["x"], s["t"], lr=1e-3)
    net.elrt_net_forward(s["x"], s["y"])
    last = net.n_layers - 1
    return loss, net.elrt_net_params(0, "dW"), net.elrt_net_params(last, "db"), net.elrt_net_params(0, "W"), s["y"]


def work(case):
    k = case["kind"]

    def local(n, p, N, extra=0, osz=4):
        nm, nin = (p + 1) ** 2, 2 * (p + 1) * N
        nu = nm * N
        return (n * (8.0 * (nm + 1) + osz * (nin + nm + extra) * nin), n * (2.0 / 3.0 * nu ** 3 + 2.0 * nu * nu * nin))

    def skel(n, p, N, osz=4):
        nm, nin = (p + 1) ** 2, 2 * (p + 1) * N
        return n * (osz * (nin + nm) * nin + 8.0 * (nin + nm)), 2.0 * n * (nin + nm) * nin

    if k == "build":
        b, f = local(case["E"], case["p"], case["N"])
    elif k == "emission":
        nu = (case["p"] + 1) ** 2 * case["N"]
        b, f = local(case["E"], case["p"], case["N"], nu)
        b += case["E"] * 8.0 * (2 * nu + nu / 8)
    elif k in ("unit", "skeleton"):
        n, osz = case["nx"] * case["nz"], 8 if k == "unit" else 4
        b, f = skel(n, case["p"], case["N"], osz)
        if k == "unit":
            b, f = b + local(n, case["p"], case["N"], 0, 8)[0], f + local(n, case["p"], case["N"])[1]
    elif k == "batch":
        b = f = 0.0
        for p in (4, 6, 8):
            n = case["nx%d" % p] * case["nz%d" % p]
            b, f = b + n * 8.0 * (2 * (p + 1) ** 2 + 1), f + local(n, p, case["N"])[1] + skel(n, p, case["N"])[1]
    else:
        nm, nin = (case["p"] + 1) ** 2, 2 * (case["p"] + 1) * case["N"]
        nout, w, h = (nin + nm) * nin, case["width"], case["hidden"]
        par = (nm + 1) * w + (h - 1) * w * w + w * nout
        if k == "infer":
            b, f = 4.0 * par + case["E"] * (8.0 * (nm + 2) + 4.0 * nout), 2.0 * par * case["E"]
        else:  # weights and both moments read and written, gradients written; inputs, targets and outputs once
            b, f = 28.0 * par + case["B"] * 4.0 * (2 * nout + 2 * nm), 8.0 * par * case["B"]
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------------------------- 64-bit values

class _Disc:
    """Directions, phase matrix and face maps of a discretisation, from their definitions."""

    def __init__(self, p, N, hg):
        n1, dth, half = p + 1, 2.0 * math.pi / N, N // 2
        x, w, D = _lgl(p)
        k = np.arange(N)
        sx, sz = (np.sin((k + 1) * dth) - np.sin(k * dth)) / dth, (np.cos(k * dth) - np.cos((k + 1) * dth)) / dth
        gx, gw = np.polynomial.legendre.leggauss(64)

        def hg_p(t):
            return (1.0 - hg * hg) / (1.0 + hg * hg - 2.0 * hg * np.cos(t)) ** 1.5
        t = 0.5 * dth * (gx + 1.0)
        W = np.array([[gw @ hg_p((a - b) * dth + t[:, None] - t[None, :]) @ gw for b in k] for a in k])
        W /= W.sum(axis=1, keepdims=True)
        nodes = [np.arange(n1), p + n1 * np.arange(n1), np.arange(n1) + n1 * p, n1 * np.arange(n1)]
        sn = [-sz, sx, sz, -sx]
        rows, cols, val = [], [], []
        for F in range(4):
            out, inc = [q for q in k if sn[F][q] > 0], [q for q in k if sn[F][q] < 0]
            for m in range(n1):
                rows += [q * n1 * n1 + nodes[F][m] for q in out]
                cols += [q * n1 * n1 + nodes[F][m] for q in inc]
                val += [-w[m] * sn[F][q] for q in inc]
        nm = n1 * n1
        w2 = np.outer(w, w).reshape(-1)
        Gx, Gz = np.kron(np.eye(n1), D), np.kron(D, np.eye(n1))
        T = np.zeros((N, nm, nm))  # transport of angle q without absorption
        for q in range(N):
            T[q] = -(sx[q] * Gx + sz[q] * Gz).T * w2[None, :]
            for F in range(4):
                if sn[F][q] > 0:
                    for m in range(n1):
                        T[q, nodes[F][m], nodes[F][m]] += w[m] * sn[F][q]

        def dev(a):
            return torch.tensor(np.asarray(a), device=DEV)
        self.nm, self.N, self.nu, self.nf, self.nin, self.half, self.n1 = nm, N, nm * N, n1 * half, 4 * n1 * half, half, n1
        self.T, self.W, self.w2 = dev(T), dev(W), dev(w2)
        self.rows, self.cols, self.val = dev(rows), dev(cols), dev(val)

    def solve(self, kh, om, src=None):
        """X (and f_u) of a chunk of elements by block elimination, one angular cell a block (the matrices need no pivoting)."""
        n, N, nm = kh.shape[0], self.N, self.nm
        A = torch.zeros(n, N, nm, N, nm, device=DEV, dtype=torch.float64)
        m = self.w2 * kh
        i = torch.arange(nm, device=DEV)
        for q in range(N):
            A[:, q, :, q, :] = self.T[q]
            A[:, q, i, q, i] += m
            for r in range(N):
                A[:, q, i, r, i] -= self.W[q, r] * om[:, None] * m
        A = A.reshape(n, self.nu, self.nu)
        nr = self.nin + (src is not None)
        B = torch.zeros(n, self.nu, nr, device=DEV, dtype=torch.float64)
        B[:, self.cols, torch.arange(self.nin, device=DEV)] = self.val
        if src is not None:
            B[:, :, -1] = (src * self.w2).reshape(n, -1)
        M = torch.cat([A, B], dim=2)
        del A, B
        inv = []
        for q in range(N):
            a, z = q * nm, (q + 1) * nm
            inv.append(torch.linalg.inv(M[:, a:z, a:z]))
            if q + 1 < N:
                M[:, z:, z:] -= M[:, z:, a:z] @ (inv[q] @ M[:, a:z, z:])
        X = M[:, :, self.nu:]
        for q in range(N - 1, -1, -1):
            a, z = q * nm, (q + 1) * nm
            X[:, a:z] = inv[q] @ (X[:, a:z] - M[:, a:z, z:self.nu] @ X[:, z:])
        return X

    def build(self, kappa, omega, h, src=None, keep=False):
        n, out = kappa.shape[0], []
        kh = kappa * (0.5 * (h[:, None] if torch.is_tensor(h) else h))
        step = max(1, int(6e9 / (8.0 * self.nu * (self.nu + self.nin))))
        for a in range(0, n, step):
            sl = slice(a, min(n, a + step))
            X = self.solve(kh[sl], omega[sl], None if src is None else src[sl] * 0.5 * h)
            c = X[:, self.rows], X.reshape(-1, self.N, self.nm, X.shape[2]).mean(dim=1)
            out.append((c[0].clone(), c[1], X.clone() if keep else None))
            del X, c
        o, m = (torch.cat([q[j] for q in out]) for j in (0, 1))
        return o, m, torch.cat([q[2] for q in out]) if keep else None

    def gather(self, nx, nz, x, g):
        """Inflow of every element: the neighbours' outflow, boundary data on the sides."""
        nf, v = self.nf, torch.zeros(nz, nx, 4, self.nf, device=DEV, dtype=torch.float64)
        x = x.reshape(nz, nx, 4, nf)
        v[1:, :, 0], v[:, :-1, 1], v[:-1, :, 2], v[:, 1:, 3] = x[:-1, :, 2], x[:, 1:, 3], x[1:, :, 0], x[:, :-1, 1]
        if g is not None:
            s = g.reshape(-1, nf)
            v[0, :, 0], v[:, -1, 1], v[-1, :, 2], v[:, 0, 3] = s[:nx], s[nx:nx + nz], s[nx + nz:2 * nx + nz], s[2 * nx + nz:]
        return v.reshape(nx * nz, -1)

    def skeleton(self, nx, nz, i2o, g, m=60):
        def ap(x):
            return x - torch.bmm(i2o, self.gather(nx, nz, x, None)[:, :, None])[:, :, 0]
        b = torch.bmm(i2o, self.gather(nx, nz, torch.zeros(nx * nz, self.nin, device=DEV, dtype=torch.float64), g)[:, :, None])[:, :, 0]
        x, nb = torch.zeros_like(b), float(b.norm())
        V = torch.zeros(m + 1, b.numel(), device=DEV, dtype=torch.float64)
        for _ in range(100):
            r = b - ap(x)
            beta = float(r.norm())
            if beta <= 1e-13 * nb:
                break
            H = np.zeros((m + 1, m))
            V[0] = r.reshape(-1) / beta
            for j in range(m):
                w = ap(V[j].reshape(b.shape)).reshape(-1)
                for _ in range(2):
                    c = V[:j + 1] @ w
                    w = w - c @ V[:j + 1]
                    H[:j + 1, j] += c.cpu().numpy()
                H[j + 1, j] = float(w.norm())
                if H[j + 1, j] <= 1e-15 * beta:
                    break
                V[j + 1] = w / H[j + 1, j]
            e = np.zeros(j + 2)
            e[0] = beta
            y = np.linalg.lstsq(H[:j + 2, :j + 1], e, rcond=None)[0]
            x = x + (torch.tensor(y, device=DEV) @ V[:j + 1]).reshape(b.shape)
        return x


def _mean(d, nx, nz, i2m, x, g):
    return torch.bmm(i2m, d.gather(nx, nz, x, g)[:, :, None])[:, :, 0]


def _act(z, act):
    return torch.nn.functional.gelu(z) if act == "gelu" else torch.nn.functional.elu(z)


def exact(case, seed):
    d, k = _inputs(case, seed), case["kind"]
    if k in ("build", "emission"):
        D = _Disc(case["p"], case["N"], 0.85)
        o, m, X = D.build(d["kappa"], d["omega"], d["h"] if d.get("h_elem") is None else d["h_elem"], d.get("source"), k == "emission")
        if k == "build":
            return o, m
        n = D.nin
        return o[:, :, :n], m[:, :, :n], o[:, :, n], m[:, :, n], X[:, :, n], X[:, :, :n]
    if k in ("unit", "skeleton"):
        D, nx, nz = _Disc(case["p"], case["N"], 0.0 if k == "unit" else 0.85), case["nx"], case["nz"]
        o, m, _ = D.build(d["kappa"], d["omega"], d["h"])
        if k == "skeleton":
            o, m = o.float().double(), m.float().double()
        x = D.skeleton(nx, nz, o, d["g"])
        return x, _mean(D, nx, nz, m, x, d["g"])
    if k == "batch":
        out = []
        for p, (nx, nz, h, kappa, omega, g) in zip((4, 6, 8), d["fields"]):
            D = _Disc(p, case["N"], 0.85)
            o, m, _ = D.build(kappa, omega, h)
            out.append(_mean(D, nx, nz, m, D.skeleton(nx, nz, o, g), g))
        return out
    W = [(a.double(), b.double()) for a, b in d["weights"]]
    if k == "infer":
        def feat(kap, om, h):
            return torch.cat([torch.log(kap * (0.5 * h)[:, None] + 1e-12), om[:, None]], dim=1)
        f = feat(*d["fit"])
        mu, sd = f.mean(dim=0), f.std(dim=0, correction=0).clamp_min(1e-3)
        x = (feat(d["kappa"], d["omega"], d["h"]) - mu) / sd
        for l, (a, b) in enumerate(W[:-1]):
            x = _act(x @ a[:, :x.shape[1]].T + b, case["act"])
        out, at = [], 0
        for lab in d["labels"]:
            n, t = lab.shape[1], lab.double()
            y = x @ W[-1][0][at:at + n].T + W[-1][1][at:at + n]
            out.append(y.mul_(t.std(dim=0, correction=0)).add_(t.mean(dim=0)))
            at += n
        nin = 2 * (case["p"] + 1) * case["N"]
        return [y.reshape(x.shape[0], -1, nin) for y in out]
    x, z, h = d["x"].double(), [], [d["x"].double()]
    for a, b in W[:-1]:
        z.append(h[-1] @ a.T + b)
        h.append(_act(z[-1], case["act"]))
    r = h[-1] @ W[-1][0].T + W[-1][1] - d["t"].double()
    loss = float(r.abs().mean())
    r = torch.sign(r) / r.numel()
    db, u = r.sum(dim=0), r @ W[-1][0]
    for l in range(len(z) - 1, -1, -1):
        if case["act"] == "gelu":
            g = 0.5 * (1.0 + torch.erf(z[l] / math.sqrt(2.0))) + z[l] * torch.exp(-0.5 * z[l] ** 2) / math.sqrt(2.0 * math.pi)
        else:
            g = torch.where(z[l] > 0, torch.ones_like(z[l]), torch.exp(z[l]))
        u = u * g
        if l:
            u = u @ W[l][0]
    return loss, u.T @ x, db, None, None  # the updated network: Adam's first step is a sign, which rounding decides near 0

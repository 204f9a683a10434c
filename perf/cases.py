"""Performance cases of the three-body eigensolver: what its users run, through its public calls.

A case is a dict of plain values with a ``kind``:

* ``apply_h``     (H - theta) psi for a block of wave functions (1D and 2D, FP64 on the FMA pipe
                  and FP64-accurate on the tensor cores);
* ``apply_prec``  (T - theta)^-1 r, the kinetic preconditioner in the solver's default arithmetic;
* ``gram``        A^T B of two column blocks (orthogonalisation, Rayleigh-Ritz matrix);
* ``update``      C = beta C + A Y (Ritz vectors, restarts, projections);
* ``train``       one loss and gradient evaluation of the warm-start network;
* ``solve``       the k lowest eigenpairs, from a cold start, default options;
* ``sweep``       a batch of independent 1D problems on concurrent streams.

The problems of the two solver kinds have well separated wanted levels (deep wells), so that the
eigenvectors, and not only the eigenvalues, are determined to well below the solver's tolerance.
"""
import math

import numpy as np
import torch

from paper_2111_02534_gb300 import tps

DTYPES = {"f64": tps.F64, "f64_tc": tps.F64_TC, "tf32_tc": tps.TF32_TC}


def listed():
    return [
        # one product on the 64 x 64 grid of the smallest workload: a user's own iteration
        # around the operator, one vector at a time; launch latency is what counts
        {"name": "apply_h_1d_n64", "kind": "apply_h", "dim": 1, "nx": 64, "ny": 64, "nvec": 1,
         "dtype": "f64", "M": 20.0, "v0": 1.0, "sigma": 1.0, "theta": 0.0},
        # the H-apply on the 512 x 512 grid of the main workload, a full block of vectors
        {"name": "apply_h_1d_n512", "kind": "apply_h", "dim": 1, "nx": 512, "ny": 512, "nvec": 8,
         "dtype": "f64_tc", "M": 40.0, "v0": 1.0, "sigma": 1.0, "theta": -0.4},
        # a grid that is square in nothing and fills no tile (coordinates with boxes of their
        # own, as in a convergence study), a short block
        {"name": "apply_h_1d_ragged", "kind": "apply_h", "dim": 1, "nx": 250, "ny": 130, "nvec": 3,
         "dtype": "f64_tc", "M": 20.0, "v0": 1.0, "sigma": 1.0, "theta": -0.4},
        # the H-apply of the 2D workload (48 points per component, 5.3 M unknowns)
        {"name": "apply_h_2d_n48", "kind": "apply_h", "dim": 2, "nx": 48, "ny": 48, "nvec": 8,
         "dtype": "f64_tc", "M": 20.0, "v0": 2.0, "sigma": 1.0, "theta": -1.0},
        # the preconditioner of the solver's correction equation on the main workload's grid
        {"name": "apply_prec_1d_n512", "kind": "apply_prec", "dim": 1, "nx": 512, "ny": 512,
         "nvec": 8, "dtype": "tf32_tc", "M": 40.0, "v0": 1.0, "sigma": 1.0, "theta": -0.4},
        # and on the 2D workload's
        {"name": "apply_prec_2d_n48", "kind": "apply_prec", "dim": 2, "nx": 48, "ny": 48, "nvec": 8,
         "dtype": "tf32_tc", "M": 20.0, "v0": 2.0, "sigma": 1.0, "theta": -1.0},
        # a search space of 16 against a block of 8 over the 2D workload's unknowns
        {"name": "gram_2d_rows", "kind": "gram", "rows": 5308416, "p": 16, "q": 8,
         "dtype": "f64_tc"},
        # Ritz vectors of a block of 8 from a search space of 36 over the rows of the main
        # workload's exchange-even sector (257 x 512)
        {"name": "update_1d_rows", "kind": "update", "rows": 131584, "p": 36, "q": 8,
         "dtype": "f64_tc", "beta": 0.0},
        # a training step of the warm-start network at its default widths
        {"name": "warmstart_train", "kind": "train", "batch": 256, "px": 32, "py": 32, "rank": 16,
         "hidden": 256},
        # the main workload's solve: 8 exchange-even pairs on the 512 x 512 grid, block 8 (with a
        # weak field on the light particle: without it some states are odd in y, and which of
        # their two equal maxima comes out positive is left to rounding)
        {"name": "solve_1d_n512", "kind": "solve", "dim": 1, "nx": 512, "ny": 512, "k": 8,
         "block": 8, "M": 40.0, "v0": 4.0, "sigma": 2.0, "field": 0.05},
        # the 2D workload's grid, one bound state, as the paper's 2D runs compute it
        {"name": "solve_2d_n48", "kind": "solve", "dim": 2, "nx": 48, "ny": 48, "k": 1, "block": 8,
         "M": 20.0, "v0": 2.0, "sigma": 1.0},
        # a parameter sweep over mass ratio and depth on grids of the four sweep sizes
        {"name": "sweep_32", "kind": "sweep", "count": 32, "k": 4, "block": 4, "nstreams": 16,
         "nmax": 384},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _even(v):
    return max(4, 2 * int(round(v / 2)))


def draw(rng):
    kind = rng.choice(["apply_h", "apply_h", "apply_h2", "prec", "prec2", "gram", "update",
                       "train", "solve", "solve2", "sweep"])
    if kind == "apply_h":
        return {"kind": "apply_h", "dim": 1, "nx": _even(_log(rng, 48, 512)),
                "ny": _even(_log(rng, 48, 512)), "nvec": int(_log(rng, 1, 12.99)),
                "dtype": rng.choice(["f64", "f64_tc", "f64_tc"]),
                "M": round(rng.uniform(1.0, 40.0), 2), "v0": round(rng.uniform(0.05, 4.0), 3),
                "sigma": rng.choice([0.5, 1.0, 2.0]), "theta": round(rng.uniform(-2.0, 0.0), 3)}
    if kind == "apply_h2":
        return {"kind": "apply_h", "dim": 2, "nx": _even(_log(rng, 12, 48)),
                "ny": _even(_log(rng, 12, 48)), "nvec": rng.randint(1, 8),
                "dtype": rng.choice(["f64", "f64_tc", "f64_tc", "f64_tc"]),
                "M": round(rng.uniform(5.0, 30.0), 2), "v0": round(rng.uniform(0.5, 4.0), 3),
                "sigma": 1.0, "theta": round(rng.uniform(-2.0, 0.0), 3)}
    if kind == "prec":
        return {"kind": "apply_prec", "dim": 1, "nx": _even(_log(rng, 48, 512)),
                "ny": _even(_log(rng, 48, 512)), "nvec": int(_log(rng, 1, 12.99)),
                "dtype": "tf32_tc", "M": round(rng.uniform(1.0, 40.0), 2), "v0": 1.0,
                "sigma": 1.0, "theta": round(rng.uniform(-2.0, -0.1), 3)}
    if kind == "prec2":
        return {"kind": "apply_prec", "dim": 2, "nx": 4 * int(_log(rng, 3, 12.99)),
                "ny": 4 * int(_log(rng, 3, 12.99)), "nvec": rng.randint(1, 8),
                "dtype": "tf32_tc", "M": round(rng.uniform(5.0, 30.0), 2), "v0": 1.0,
                "sigma": 1.0, "theta": round(rng.uniform(-2.0, -0.1), 3)}
    if kind in ("gram", "update"):
        rows = int(_log(rng, 1.0e4, 5.3e6))
        q = rng.randint(1, 8)
        p = max(q, int(_log(rng, 2, min(64.99, 1.3e8 / rows))))
        c = {"kind": kind, "rows": rows, "p": p, "q": q,
             "dtype": rng.choice(["f64", "f64_tc", "f64_tc"])}
        if kind == "update":
            c["beta"] = rng.choice([0.0, 1.0])
        return c
    if kind == "train":
        return {"kind": "train", "batch": int(_log(rng, 32, 512)), "px": rng.choice([16, 24, 32]),
                "py": rng.choice([16, 32]), "rank": rng.choice([8, 16]),
                "hidden": rng.choice([128, 256])}
    if kind == "solve":
        return {"kind": "solve", "dim": 1, "nx": _even(_log(rng, 96, 512)),
                "ny": _even(_log(rng, 128, 512)), "k": rng.randint(1, 4),
                "block": rng.choice([4, 6, 8]), "M": round(rng.uniform(20.0, 40.0), 2),
                "v0": round(rng.uniform(2.0, 4.0), 3), "sigma": 2.0, "field": 0.05}
    if kind == "solve2":
        return {"kind": "solve", "dim": 2, "nx": 4 * rng.randint(6, 12), "ny": 4 * rng.randint(6, 12),
                "k": 1, "block": rng.choice([4, 6, 8]), "M": round(rng.uniform(10.0, 30.0), 2),
                "v0": round(rng.uniform(1.5, 3.0), 3), "sigma": 1.0}
    return {"kind": "sweep", "count": rng.randint(8, 32), "k": rng.randint(2, 4), "block": 4,
            "nstreams": rng.choice([8, 16]), "nmax": rng.choice([192, 256, 384])}


# ------------------------------------------------------------------- inputs


def _box(case):
    """Grid sizes and half box lengths of a case, in the order of the coordinates."""
    d = case["dim"]
    return [case["nx"]] * d + [case["ny"]] * d, [20.0] * (2 * d)


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _context(case, M, v0):
    ctx = tps.Context(case["dim"], 0)
    ctx.set_masses(M, 1.0, 1.0)
    n, L = _box(case)
    ctx.set_grid(n, L)
    if case.get("field"):
        _, x = _kinetic(n, L, M)
        ctx.set_potential(_potential(x, v0, case["sigma"], case["field"]).contiguous())
    else:
        ctx.set_pair_potential(tps.GAUSS, v0, case["sigma"])
    return ctx


def _waves(n, nvec, seed):
    """nvec functions on the grid: bound-state-like bumps of several widths with a broadband
    part a thousandth their size, as search vectors and residuals have (FP64, unit norm)."""
    g = _generator(seed)
    out = torch.zeros(nvec, *n, dtype=torch.float64, device="cuda")
    for v in range(nvec):
        env = torch.ones((), dtype=torch.float64, device="cuda")
        noise = torch.ones((), dtype=torch.float64, device="cuda")
        for k, m in enumerate(n):
            x = torch.linspace(-1, 1, m + 1, dtype=torch.float64, device="cuda")[:-1]
            r = torch.rand(4, generator=g, device="cuda", dtype=torch.float64)
            bump = torch.exp(-((x - 0.6 * (r[0] - 0.5)) / (0.08 + 0.5 * r[1])) ** 2)
            bump = bump * torch.cos(12 * r[2] * x + 6 * r[3])
            shape = [1] * len(n)
            shape[k] = m
            env = env * bump.reshape(shape)
            noise = noise * torch.exp(-2 * (x / 0.7) ** 2).reshape(shape)
        out[v] = env + 1e-3 * noise * torch.randn(n, generator=g, device="cuda",
                                                  dtype=torch.float64)
        out[v] /= out[v].norm()
    return out.reshape(nvec, -1)


def _columns(rows, p, seed):
    """A column-major rows x p block (stored [p][rows]) of unit columns."""
    a = torch.randn(p, rows, generator=_generator(seed), device="cuda", dtype=torch.float64)
    return a / a.norm(dim=1, keepdim=True)


def _problem(case, seed):
    """Mass ratio and depth of a solve: the case's own, moved a little by the seed."""
    r = np.random.default_rng(seed)
    return case["M"] * (1 + 0.02 * r.random()), case["v0"] * (1 + 0.02 * r.random())


def _sweep(case, seed):
    """The instances of a sweep: (case of one solve, M, v0)."""
    r = np.random.default_rng(seed)
    sizes = [n for n in (128, 192, 256, 384) if n <= case["nmax"]]
    got = []
    for i in range(case["count"]):
        n = sizes[i % len(sizes)]
        one = {"dim": 1, "nx": n, "ny": n, "sigma": 2.0, "k": case["k"], "block": case["block"]}
        got.append((one, float(r.uniform(20, 40)), float(r.uniform(2, 4))))
    return got


def _network(case, seed):
    """Weights (He-initialised, the library's parameter order), features and targets."""
    r = np.random.default_rng(seed)
    h, out = case["hidden"], case["rank"] * (case["px"] + case["py"])
    params = []
    for a, b in ((4, h), (h, h), (h, h), (h, out)):
        params += [r.standard_normal(a * b) * math.sqrt(2.0 / a), 0.01 * r.standard_normal(b)]
    x = np.stack([r.uniform(0, 1, case["batch"]), r.uniform(-0.8, 0.3, case["batch"]),
                  r.integers(-1, 2, case["batch"]).astype(float),
                  r.integers(0, 8, case["batch"]) / 8.0], axis=1)
    t = r.standard_normal((case["batch"], case["px"], case["py"]))
    t *= np.exp(-0.2 * np.arange(case["px"]))[:, None] * np.exp(-0.2 * np.arange(case["py"]))
    return (np.concatenate(params).astype(np.float32), x.astype(np.float32), t.astype(np.float32))


TOL = 1e-12  # of ||H||, the workloads' tolerance


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind in ("apply_h", "apply_prec"):
        s["ctx"] = _context(case, case["M"], case["v0"])
        s["in"] = _waves(_box(case)[0], case["nvec"], seed)
        s["out"] = torch.empty_like(s["in"])
    elif kind == "gram":
        s["ctx"] = tps.Context(1, 0)
        s["A"] = _columns(case["rows"], case["p"], 2 * seed)
        s["B"] = _columns(case["rows"], case["q"], 2 * seed + 1)
        s["B"] += 0.5 * s["A"][:case["q"]]
        s["G"] = torch.empty(case["q"], case["p"], dtype=torch.float64, device="cuda")
    elif kind == "update":
        s["ctx"] = tps.Context(1, 0)
        s["A"] = _columns(case["rows"], case["p"], 2 * seed)
        y = torch.randn(case["p"], case["p"], generator=_generator(seed), device="cuda",
                        dtype=torch.float64)
        s["Y"] = torch.linalg.qr(y)[0][:, :case["q"]].T.contiguous()
        s["C0"] = _columns(case["rows"], case["q"], 2 * seed + 1)
        s["C"] = torch.empty_like(s["C0"])
    elif kind == "train":
        params, x, t = _network(case, seed)
        s["model"] = tps.WarmStart(case["px"], case["py"], case["rank"], case["hidden"])
        s["model"].set_params(params)
        s["X"], s["T"] = torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()
    elif kind == "solve":
        s["ctx"] = _context(case, *_problem(case, seed))
        s["evecs"] = torch.empty(case["k"], math.prod(_box(case)[0]), dtype=torch.float64,
                                 device="cuda")
    else:
        got = _sweep(case, seed)
        s["ctxs"] = [_context(one, M, v0) for one, M, v0 in got]
        s["evecs"] = [torch.empty(case["k"], one["nx"] * one["ny"], dtype=torch.float64,
                                  device="cuda") for one, _, _ in got]
    return s


# --------------------------------------------------------------------- runs


def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "apply_h":
        s["ctx"].apply_h(s["in"], s["out"], theta=c["theta"], dtype=DTYPES[c["dtype"]])
        return s["out"]
    if kind == "apply_prec":
        s["ctx"].apply_prec(s["in"], s["out"], c["theta"], dtype=DTYPES[c["dtype"]])
        return s["out"]
    if kind == "gram":
        s["ctx"].gram(s["A"], c["p"], s["B"], c["q"], c["rows"], s["G"], dtype=DTYPES[c["dtype"]])
        return s["G"]
    if kind == "update":
        if c["beta"]:
            s["C"].copy_(s["C0"])
        s["ctx"].block_update(s["A"], c["p"], s["Y"], c["q"], c["beta"], s["C"], c["rows"],
                              dtype=DTYPES[c["dtype"]])
        return s["C"]
    if kind == "train":
        loss, grad = s["model"].loss_grad(s["X"], s["T"], want_grad=True)
        return {"loss": loss, "grad": grad}
    if kind == "solve":
        lam, _ = s["ctx"].solve(c["k"], tps.X_EVEN if c["dim"] == 1 else tps.ANY, TOL, c["block"],
                                s["evecs"])
        return {"lam": lam, "evecs": s["evecs"]}
    lam, _, status = tps.solve_batch(s["ctxs"], [c["k"]] * c["count"], tps.X_EVEN, TOL, c["block"],
                                     s["evecs"], nstreams=c["nstreams"])
    return {"lam": np.stack(lam), "status": np.array(status),
            "evecs": torch.cat([e.reshape(-1) for e in s["evecs"]])}


def work(case):
    """Bytes and operations of one pass: each input read and each output written once; the dense
    mode products of the scheme (a preconditioner has two of them per mode)."""
    kind = case["kind"]
    if kind in ("apply_h", "apply_prec", "solve"):
        n, _ = _box(case)
        N = math.prod(n)
        if kind == "apply_h":
            return {"bytes": 8 * N * (2 * case["nvec"] + 1),
                    "flops": case["nvec"] * (2 * N * sum(n) + 3 * N)}
        if kind == "apply_prec":
            return {"bytes": 16 * N * case["nvec"], "flops": case["nvec"] * (4 * N * sum(n) + N)}
        return _solve_work(N // (2 if case["dim"] == 1 else 1), sum(n), case["k"], case["block"])
    if kind == "gram":
        return {"bytes": 8 * case["rows"] * (case["p"] + case["q"]),
                "flops": 2 * case["rows"] * case["p"] * case["q"]}
    if kind == "update":
        return {"bytes": 8 * case["rows"] * (case["p"] + case["q"] * (3 if case["beta"] else 1)),
                "flops": 2 * case["rows"] * case["p"] * case["q"]}
    if kind == "train":
        h, out = case["hidden"], case["rank"] * (case["px"] + case["py"])
        weights = 4 * h + 2 * h * h + h * out
        contraction = 6 * case["rank"] * case["px"] * case["py"]
        return {"bytes": 8 * weights + 4 * case["batch"] * (4 + case["px"] * case["py"]),
                "flops": case["batch"] * (6 * weights + contraction)}
    total = {"bytes": 0, "flops": 0}
    for one, _, _ in _sweep(case, 0):
        w = _solve_work(one["nx"] * one["ny"] // 2, one["nx"] + one["ny"], case["k"], case["block"])
        total = {k: total[k] + w[k] for k in total}
    return total


def _solve_work(N, modes, k, block):
    """About ten outer iterations: an H and a preconditioner application of a block, and two
    passes over a search space of twice the block, each."""
    b = max(block, k)
    return {"bytes": 10 * (8 * N * 4 * b + 2 * 8 * N * 2 * b),
            "flops": 10 * b * (6 * N * modes + 4 * N * 2 * b)}


# -------------------------------------------------- the same in 64 bits, plainly


def _kinetic(n, L, M):
    """Eigenvalues of T on the Fourier grid, in torch's FFT order, and the coordinates."""
    d = len(n) // 2
    a = [-1.0 / M] * d + [-(2 * M + 1) / (4 * M)] * d
    T = torch.zeros((), dtype=torch.float64, device="cuda")
    x = []
    for k, (m, l) in enumerate(zip(n, L)):
        w = torch.fft.fftfreq(m, d=1.0 / m, dtype=torch.float64, device="cuda") * (math.pi / l)
        shape = [1] * len(n)
        shape[k] = m
        T = T - a[k] * (w * w).reshape(shape)
        x.append((-l + 2 * l / m * torch.arange(m, dtype=torch.float64,
                                                device="cuda")).reshape(shape))
    return T, x


def _potential(x, v0, sigma, field=0.0):
    """The pair potential of the problem, and with it a field on the light particle (1D)."""
    d = len(x) // 2
    V = field * torch.sin(math.pi / 20.0 * x[-1]) if field else 0
    for sign in (-1, 1):
        r2 = sum((x[d + k] + sign * 0.5 * x[k]) ** 2 for k in range(d))
        V = V - v0 * torch.exp(-r2 / sigma ** 2)
    return V


def _spectral(v, n, f):
    """Every function of a [m, N] block with its Fourier coefficients multiplied by f."""
    out = torch.empty_like(v)
    for i in range(v.shape[0]):
        w = torch.fft.fftn(v[i].reshape(n))
        out[i] = torch.fft.ifftn(w * f).real.reshape(-1)
    return out


def _lowest(case, M, v0, k):
    """The k lowest (1D: x-even) eigenpairs by a plain block Davidson method."""
    n, L = _box(case)
    T, x = _kinetic(n, L, M)
    V = _potential(x, v0, case["sigma"], case.get("field", 0.0)).reshape(-1)

    def even(v):
        if case["dim"] != 1:
            return v
        w = v.reshape(-1, *n)
        return (0.5 * (w + torch.roll(w.flip(1), 1, 1))).reshape(v.shape)

    b = k + 3
    N = math.prod(n)
    X = torch.randn(b, N, generator=_generator(1), device="cuda", dtype=torch.float64)
    Q = torch.linalg.qr(even(_spectral(X, n, 1.0 / (T + 1.0) ** 2)).T)[0]
    HQ = (_spectral(Q.T.contiguous(), n, T) + V * Q.T).T
    scale = float(T.max())
    for _ in range(120):
        lam, y = torch.linalg.eigh(0.5 * (Q.T @ HQ + HQ.T @ Q))
        lam, y = lam[:b], y[:, :b]
        X, R = Q @ y, HQ @ y - (Q @ y) * lam
        worst = float(R[:, :k].norm(dim=0).max())
        if worst < 2e-15 * scale:
            break
        if Q.shape[1] + b > 8 * b:
            keep = torch.linalg.qr(torch.cat([X, Q[:, -b:]], 1))[0]
            Q = keep
            HQ = (_spectral(Q.T.contiguous(), n, T) + V * Q.T).T
        shift = 0.05 + 1.02 * abs(float(lam[0]))
        t = even(_spectral(R.T.contiguous(), n, 1.0 / (T + shift))).T
        for _ in range(2):
            t = t - Q @ (Q.T @ t)
            t = torch.linalg.qr(t)[0]
        Q = torch.cat([Q, t], 1)
        HQ = torch.cat([HQ, (_spectral(t.T.contiguous(), n, T) + V * t.T).T], 1)
    X = X[:, :k].T.contiguous()
    X = X / X.norm(dim=1, keepdim=True)
    top = X.gather(1, X.abs().argmax(1, keepdim=True))
    return lam[:k].cpu().numpy(), X * torch.sign(top)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("apply_h", "apply_prec"):
        n, L = _box(case)
        T, x = _kinetic(n, L, case["M"])
        v = _waves(n, case["nvec"], seed)
        if kind == "apply_prec":
            return _spectral(v, n, 1.0 / (T - case["theta"]))
        V = _potential(x, case["v0"], case["sigma"]).reshape(-1)
        return _spectral(v, n, T) + (V - case["theta"]) * v
    if kind == "gram":
        A = _columns(case["rows"], case["p"], 2 * seed)
        B = _columns(case["rows"], case["q"], 2 * seed + 1)
        return (B + 0.5 * A[:case["q"]]) @ A.T
    if kind == "update":
        A = _columns(case["rows"], case["p"], 2 * seed)
        y = torch.randn(case["p"], case["p"], generator=_generator(seed), device="cuda",
                        dtype=torch.float64)
        Y = torch.linalg.qr(y)[0][:, :case["q"]]
        C = _columns(case["rows"], case["q"], 2 * seed + 1)
        return case["beta"] * C + (A.T @ Y).T.contiguous()
    if kind == "train":
        params, x, t = (torch.from_numpy(v).double() for v in _network(case, seed))
        params.requires_grad_(True)
        a, at, h, r = x, 0, case["hidden"], case["rank"]
        widths = [4, h, h, h, r * (case["px"] + case["py"])]
        for i in range(4):
            m, o = widths[i], widths[i + 1]
            z = a @ params[at:at + m * o].reshape(m, o) + params[at + m * o:at + m * o + o]
            at += m * o + o
            a = torch.nn.functional.gelu(z) if i < 3 else z
        C = a[:, :r * case["px"]].reshape(-1, r, case["px"])
        D = a[:, r * case["px"]:].reshape(-1, r, case["py"])
        P = torch.einsum("bra,brc->bac", C, D)
        loss = (1 - (P * t).sum((1, 2)) ** 2 / ((P * P).sum((1, 2)) * (t * t).sum((1, 2)))).mean()
        loss.backward()
        return {"loss": float(loss), "grad": params.grad.numpy()}
    if kind == "solve":
        lam, X = _lowest(case, *_problem(case, seed), case["k"])
        return {"lam": lam, "evecs": X}
    got = [_lowest(one, M, v0, case["k"]) for one, M, v0 in _sweep(case, seed)]
    return {"lam": np.stack([g[0] for g in got]), "status": None,
            "evecs": torch.cat([g[1].reshape(-1) for g in got])}

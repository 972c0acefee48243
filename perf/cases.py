"""The framework's work as users have it done: what is timed, on which inputs, and what 64 bits make of it.

A case is one call (or one call and its backward) of the binding in
``paper_2604_02917_gb300.mv`` on a seeded synthetic panel:

* ``solve``       NPGA to a KKT residual of 1e-6 from a kept ``Solver`` (full, compressed or explicit-Sigma model)
* ``refined``     the same on a BF16 or FP8 copy, finished on the FP32 factor
* ``frontier``    many return targets on one low-precision factor
* ``batch``       independent problems of uneven size in one call
* ``adjoint``     a fixed number of iterations through autograd, forward and backward
* ``center``      mean, factor and trace from a return panel
* ``sigma``       the explicit covariance from the factor
* ``sketch``      the Gaussian sketch of the factor
* ``countsketch`` the sparse sketch of the factor
* ``truncate``    rank-k factor and ridge from a sketch

Inputs come from the factor model of the repository's workloads (Gaussian
loadings, Student-t(4) factors, Gaussian noise, a drift per asset), drawn and
centred on the GPU with plain torch, so that they do not depend on the code
that is measured.
"""
import math

import numpy as np
import torch

from paper_2604_02917_gb300 import mv

F64 = torch.float64
DEV = "cuda"
ESIZE = {"f32": 4, "bf16": 2, "fp8": 1}
ITERS = 50      # iterations that a solve to 1e-6 takes at the full shape (more on small panels): used by work() alone
N_FULL, T_FULL = 5440, 48374


def listed():
    return [
        # The full model at the real-data shape (5440 A-shares, 48374 five-minute periods): the framework's headline solve.
        {"name": "solve_full_f32", "kind": "solve", "n": N_FULL, "T": T_FULL, "dtype": "f32", "layout": "tn", "steps": 25,
         "lanczos": True, "factors": 20, "vol_lo": 0.01, "vol_hi": 0.03},
        # A desk-sized universe of 200 assets in the default layout with default options: launches and latency.
        {"name": "solve_small_f32", "kind": "solve", "n": 200, "T": 1000, "dtype": "f32", "layout": "nt", "steps": 50,
         "lanczos": False, "factors": 5, "vol_lo": 0.005, "vol_hi": 0.02},
        # The compressed (sketch-truncate-ridge) model of the full universe, rank 512: many solves on one small factor.
        {"name": "solve_str_512", "kind": "solve", "n": N_FULL, "T": 512, "dtype": "f32", "layout": "str", "steps": 25,
         "lanczos": True, "factors": 20, "vol_lo": 0.01, "vol_hi": 0.03},
        # An odd mid-sized universe whose products stream a BF16 copy, finished on the FP32 factor.
        {"name": "refined_bf16_mid", "kind": "refined", "n": 1733, "T": 9001, "dtype": "bf16", "layout": "tn", "steps": 25,
         "factors": 10, "vol_lo": 0.005, "vol_hi": 0.02},
        # A 64-point efficient frontier of the full universe on one BF16 factor.
        {"name": "frontier_64_bf16", "kind": "frontier", "n": N_FULL, "T": T_FULL, "dtype": "bf16", "targets": 64, "steps": 25,
         "factors": 20, "vol_lo": 0.01, "vol_hi": 0.03},
        # Independent universes of uneven size (500..5000 assets, 2000..20000 periods) solved in one call.
        {"name": "batch_32_uneven", "kind": "batch", "count": 32, "n_lo": 500, "n_hi": 5000, "T_lo": 2000, "T_hi": 20000,
         "sizes": 1000,
         "dtype": "f32", "layout": "tn", "steps": 50},
        # A portfolio layer inside a training step: 500 unrolled iterations, forward and backward, taped as one segment (the tape is small beside the memory).
        {"name": "adjoint_2000", "kind": "adjoint", "n": 2000, "T": 10000, "iters": 500, "every": 512},
        # Mean, centred factor (transposed, as the solve wants it) and trace of the full panel.
        {"name": "center_full_f32", "kind": "center", "n": N_FULL, "T": T_FULL, "dtype": "f32", "layout": "tn"},
        # The classical model: the explicit covariance of the full panel.
        {"name": "sigma_full_f32", "kind": "sigma", "n": N_FULL, "T": T_FULL, "dtype": "f32"},
        # The Gaussian sketch of the full BF16 factor to 8192 columns, first step of the compressed model.
        {"name": "sketch_full_bf16", "kind": "sketch", "n": N_FULL, "T": T_FULL, "m": 8192, "dtype": "bf16"},
        # The sparse sketch of the full factor to the same width.
        {"name": "countsketch_full_f32", "kind": "countsketch", "n": N_FULL, "T": T_FULL, "m": 8192, "dtype": "f32", "layout": "tn"},
        # Truncation of a mid-sized sketch to rank 128 with the default ridge.
        {"name": "truncate_2500", "kind": "truncate", "n": 2500, "m": 4096, "k": 128},
    ]


def _log(rng, lo, hi):
    """A whole number between lo and hi, even over the logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _panel(rng, n_lo, n_hi, T_lo, T_hi, most=N_FULL * T_FULL):
    n = _log(rng, n_lo, n_hi)
    return n, _log(rng, T_lo, max(T_lo, min(T_hi, most // n)))


def draw(rng):
    kind = rng.choice(["solve", "solve", "compressed", "explicit", "refined", "frontier", "batch", "adjoint", "center", "center",
                       "sigma", "sketch", "countsketch", "truncate"])
    vol = {"factors": rng.randint(3, 20), "vol_lo": 0.005 if rng.random() < 0.5 else 0.01}
    vol["vol_hi"] = 4 * vol["vol_lo"] if vol["vol_lo"] < 0.01 else 0.03
    if kind == "solve":
        n, T = _panel(rng, 200, 8000, 1000, T_FULL)
        lanczos = rng.random() < 0.6
        return {"kind": "solve", "n": n, "T": T, "dtype": rng.choice(["f32", "f32", "bf16", "fp8"]), "layout": rng.choice(["tn", "tn", "nt"]),
                "steps": 25 if lanczos else 50, "lanczos": lanczos, **vol}
    if kind == "compressed":
        return {"kind": "solve", "n": _log(rng, 500, N_FULL), "T": _log(rng, 32, 512), "dtype": "f32", "layout": "str", "steps": 25, "lanczos": True, **vol}
    if kind == "explicit":
        n = _log(rng, 200, N_FULL)
        return {"kind": "solve", "n": n, "T": _log(rng, max(1000, n), 16000), "dtype": "f32", "layout": "sigma", "steps": 50, "lanczos": False, **vol}
    if kind == "refined":
        n, T = _panel(rng, 200, N_FULL, 1000, T_FULL)
        return {"kind": "refined", "n": n, "T": T, "dtype": rng.choice(["bf16", "fp8"]), "layout": rng.choice(["tn", "nt"]), "steps": 25, **vol}
    if kind == "frontier":
        n, T = _panel(rng, 200, N_FULL, 1000, T_FULL)
        return {"kind": "frontier", "n": n, "T": T, "dtype": rng.choice(["bf16", "bf16", "fp8"]), "targets": _log(rng, 4, 64), "steps": 25, **vol}
    if kind == "batch":
        n_hi, T_hi = _log(rng, 600, 5000), _log(rng, 3000, 20000)
        return {"kind": "batch", "count": _log(rng, 2, 24), "n_lo": rng.randint(200, 500), "n_hi": n_hi, "T_lo": 2000, "T_hi": T_hi, "sizes": rng.randint(0, 9999),
                "dtype": "f32", "layout": rng.choice(["tn", "tn", "nt"]), "steps": 50}
    if kind == "adjoint":
        return {"kind": "adjoint", "n": _log(rng, 200, 2000), "T": _log(rng, 500, 10000), "iters": rng.randint(60, 400), "every": 512}
    if kind == "center":
        n, T = _panel(rng, 200, 8000, 500, 60000)
        return {"kind": "center", "n": n, "T": T, "dtype": rng.choice(["f32", "f32", "bf16", "fp8"]), "layout": rng.choice(["tn", "nt"])}
    if kind == "sigma":
        n, T = _panel(rng, 300, N_FULL, 1000, T_FULL)
        return {"kind": "sigma", "n": n, "T": T, "dtype": rng.choice(["f32", "f32", "bf16", "fp8"])}
    if kind == "sketch":
        n, T = _panel(rng, 300, N_FULL, 1000, T_FULL)
        return {"kind": "sketch", "n": n, "T": T, "m": _log(rng, 200, 4096), "dtype": rng.choice(["bf16", "bf16", "f32", "fp8"])}
    if kind == "countsketch":
        n, T = _panel(rng, 300, N_FULL, 1000, T_FULL)
        return {"kind": "countsketch", "n": n, "T": T, "m": _log(rng, 200, 8192), "dtype": rng.choice(["f32", "f32", "bf16", "fp8"]),
                "layout": rng.choice(["tn", "tn", "nt"])}
    n, m = _log(rng, 300, 2500), _log(rng, 500, 4096)
    return {"kind": "truncate", "n": n, "m": m, "k": min(_log(rng, 16, 128), n // 4, m // 4)}


# ------------------------------------------------------------------ inputs


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _returns(g, n, T, factors=5, vol_lo=0.005, vol_hi=0.02):
    """An n x T FP32 return panel of the factor model."""
    B = 0.01 * torch.randn((n, factors), generator=g, device=DEV)
    chi = torch.randn((4, factors, T), generator=g, device=DEV).square().sum(0)
    f = (0.01 / math.sqrt(2.0)) * torch.randn((factors, T), generator=g, device=DEV) / torch.sqrt(chi / 4)
    vol = vol_lo + (vol_hi - vol_lo) * torch.rand((n, 1), generator=g, device=DEV)
    drift = -2e-4 + 8e-4 * torch.rand((n, 1), generator=g, device=DEV)
    R = torch.randn((n, T), generator=g, device=DEV)
    return R.mul_(vol).addmm_(B, f).add_(drift)


def _centred(R):
    """(mu, L) of a panel in 64 bits."""
    mu = R.sum(1, dtype=F64) / R.shape[1]
    return mu, (R - mu[:, None]) / math.sqrt(R.shape[1] - 1)


def _stored(L, dtype, layout):
    """(tensor, row scales) of the 64-bit n x T factor as the framework stores it, its leading dimension padded with zeros."""
    scale = None
    if dtype == "fp8":
        scale = (L.abs().amax(1) / 448).clamp_min(1e-30).float()
        L = (L / scale[:, None]).float().clamp(-448, 448)
    if layout == "tn":
        L = L.T
    pad = mv.padded_ld(L.shape[1], mv.DTYPES[dtype])
    kind = {"f32": torch.float32, "bf16": torch.bfloat16, "fp8": torch.float8_e4m3fn}[dtype]
    out = torch.zeros((L.shape[0], pad), dtype=torch.uint8 if dtype == "fp8" else kind, device=DEV)
    out[:, :L.shape[1]] = L.to(kind).view(torch.uint8) if dtype == "fp8" else L
    return out, scale


def _wide(L, scale, dtype, layout, n, T):
    """The stored factor as an n x T matrix in 64 bits."""
    if dtype == "fp8":
        L = L.view(torch.float8_e4m3fn).float()
    L = (L[:T, :n].T if layout == "tn" else L[:n, :T]).to(F64)
    return L if scale is None else L * scale[:, None].to(F64)


def _target(mu, q=0.6):
    return float(torch.quantile(mu, q))


def _problem(case, seed):
    """Factor (as stored), mean and target of a solve, and what its options are."""
    c, g = case, _gen(seed)
    n, T = c["n"], c["T"]
    d = {"gamma": 0.0}
    if c["layout"] == "str":  # U diag(sigma), the head of a sketch's flat spectrum, and its ridge
        mu = -2e-4 + 8e-4 * torch.rand(n, generator=g, device=DEV, dtype=F64)
        s = c["vol_hi"] * torch.linspace(1.2, 0.9, T, device=DEV, dtype=F64)
        L = torch.linalg.qr(torch.randn((n, T), generator=g, device=DEV, dtype=torch.float32))[0].to(F64) * s
        d["gamma"] = 1e-4 * (0.5 * (c["vol_lo"] + c["vol_hi"])) ** 2
        d["L"], d["scale"] = _stored(L, "f32", "nt")
    else:
        R = _returns(g, n, T, c["factors"], c["vol_lo"], c["vol_hi"])
        mu, L = _centred(R)
        del R
        if c["layout"] == "sigma":
            d["L"], d["scale"] = _stored((L.float() @ L.float().T).to(F64), "f32", "nt")
        else:
            d["L"], d["scale"] = _stored(L, c["dtype"], c["layout"])
    if c["kind"] == "refined":
        d["L_hi"], _ = _stored(L, "f32", "tn")
    d["mu"], d["target"] = mu, _target(mu)
    d["start"] = torch.randn(n, generator=g, device=DEV, dtype=F64)
    return d


def _batch_sizes(case):
    r = np.random.default_rng(case["sizes"])
    return list(zip(r.integers(case["n_lo"], case["n_hi"] + 1, case["count"]).tolist(), r.integers(case["T_lo"], case["T_hi"] + 1, case["count"]).tolist()))


def _batch_problem(case, seed, j, n, T):
    g = _gen(seed * 1009 + j)
    R = _returns(g, n, T)
    mu, L = _centred(R)
    L, _ = _stored(L, case["dtype"], case["layout"])
    return {"L": L, "mu": mu, "R_target": _target(mu), "T": T, "layout": case["layout"],
            "power_start": torch.randn(n, generator=g, device=DEV, dtype=F64)}


def _frontier_targets(mu, count):
    return torch.linspace(_target(mu, 0.1), _target(mu, 0.9), count, dtype=F64, device=DEV)


def _adjoint_inputs(case, seed):
    g = _gen(seed)
    mu, L = _centred(_returns(g, case["n"], case["T"]))
    w = torch.randn(case["n"], generator=g, device=DEV, dtype=F64)
    return _stored(L, "f32", "nt")[0], mu, _target(mu), w


def _sketch_inputs(case, seed):
    g = _gen(seed)
    n, T, m = case["n"], case["T"], case["m"]
    _, L = _centred(_returns(g, n, T))
    L, scale = _stored(L, case["dtype"], case.get("layout", "nt"))
    if case["kind"] == "countsketch":
        h = torch.randint(0, m, (T,), generator=g, device=DEV, dtype=torch.int32)
        return L, scale, (h, (2 * torch.randint(0, 2, (T,), generator=g, device=DEV) - 1).to(torch.int8))
    Phi = torch.zeros((m, (T + 7) // 8 * 8), dtype=torch.bfloat16, device=DEV)
    Phi[:, :T] = torch.randn((m, T), generator=g, device=DEV) / math.sqrt(m)
    return L, scale, Phi


def _sketched(case, seed):
    """A sketch of a centred panel has Gaussian columns with the panel's covariance."""
    g = _gen(seed)
    n, m = case["n"], case["m"]
    vol = 0.01 + 0.02 * torch.rand((n, 1), generator=g, device=DEV)
    B = 0.01 * 0.01 * torch.randn((n, 20), generator=g, device=DEV)
    X = torch.randn((n, m), generator=g, device=DEV).mul_(vol).addmm_(B, torch.randn((20, m), generator=g, device=DEV))
    return X.div_(math.sqrt(m)), float(vol.square().sum() + B.square().sum())


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "solve":
        d = _problem(c, seed)
        layout = "nt" if c["layout"] == "str" else c["layout"]
        return c, mv.Solver(d["L"], d["mu"], d["target"], c["T"], d["gamma"], c["dtype"], d["scale"], power_start=d["start"], layout=layout, eps=1e-6,
                            lanczos=int(c["lanczos"]), power_iters=c["steps"])
    if kind == "refined":
        d = _problem(c, seed)
        return c, mv.RefinedSolver(d["L"], d["L_hi"], d["mu"], d["target"], c["T"], dtype=c["dtype"], row_scale=d["scale"], power_start=d["start"],
                                   layout=c["layout"], layout_hi="tn", eps_lo=1e-5, eps=1e-6, lanczos=1, power_iters=c["steps"])
    if kind == "frontier":
        d = _problem(dict(c, layout="nt"), seed)
        return c, mv.FrontierSolver(d["L"], d["mu"], _frontier_targets(d["mu"], c["targets"]), c["T"], power_start=d["start"], dtype=c["dtype"],
                                    row_scale=d["scale"], eps=1e-6, lanczos=1, power_iters=c["steps"])
    if kind == "batch":
        return c, mv.BatchSolver([_batch_problem(c, seed, j, n, T) for j, (n, T) in enumerate(_batch_sizes(c))], c["dtype"], eps=1e-6, power_iters=c["steps"])
    if kind == "adjoint":
        L, mu, target, w = _adjoint_inputs(c, seed)
        return c, L.requires_grad_(), mu.requires_grad_(), target, w
    if kind == "center":
        return c, _returns(_gen(seed), c["n"], c["T"], 20, 0.01, 0.03)
    if kind == "sigma":
        return c, *_sketch_inputs(dict(c, m=1), seed)[:2]
    if kind in ("sketch", "countsketch"):
        return c, *_sketch_inputs(c, seed)
    return c, *_sketched(c, seed)


# ------------------------------------------------------------------ the calls


def run(state):
    c, kind = state[0], state[0]["kind"]
    if kind in ("solve", "refined"):
        x, info = state[1].solve()
        return {"x": x, "objective": info["objective"], "iterations": info["iterations"]}
    if kind == "frontier":
        X, infos = state[1].solve()
        return {"X": X, "objective": np.array([i["objective"] for i in infos]), "iterations": np.array([i["iterations"] for i in infos])}
    if kind == "batch":
        xs, infos = state[1].solve()
        return {"x": xs, "objective": np.array([i["objective"] for i in infos]), "iterations": np.array([i["iterations"] for i in infos])}
    if kind == "adjoint":
        _, L, mu, target, w = state
        x = mv.NPGAFunction.apply(L, mu, target, c["T"], c["iters"], 0.0, c["every"])
        dL, dmu = torch.autograd.grad(x, (L, mu), w)
        return {"x": x.detach(), "dL": dL[:, :c["T"]], "dmu": dmu}  # the padding of the leading dimension is nobody's
    if kind == "center":
        L, scale, mu, trace = mv.center_factor(state[1], c["dtype"], layout=c["layout"])
        return {"L": L, "mu": mu, "trace": trace, **({} if scale is None else {"scale": scale})}
    if kind == "sigma":
        return mv.sigma_form(state[1], c["T"], c["dtype"], state[2])
    if kind == "sketch":
        _, L, scale, Phi = state
        return mv.sketch(L, c["T"], Phi) if c["dtype"] == "bf16" else mv.sketch_dtype(L, c["T"], Phi, c["dtype"], scale)
    if kind == "countsketch":
        _, L, scale, (h, sign) = state
        return mv.countsketch(L, c["n"], c["T"], h, sign, c["m"], c["dtype"], scale, c["layout"])
    L_eff, sigma, gamma = mv.str_truncate(state[1], c["k"], -1.0, state[2])
    return {"L_eff": L_eff, "sigma": sigma, "gamma": gamma}


def work(case):
    """Factor bytes once per product (both half-products share one read), inputs and outputs once; two multiply-adds per entry and product."""
    c, kind = case, case["kind"]
    if kind == "batch":
        e = (c["n_lo"] + c["n_hi"]) / 2 * (c["T_lo"] + c["T_hi"]) / 2 * c["count"]
        p = c["steps"] + 2 * ITERS
        return {"bytes": e * ESIZE[c["dtype"]] * p, "flops": 4 * e * p}
    n, T = c["n"], c.get("T", 1)
    e = float(n) * T
    if kind == "solve" and c["layout"] == "sigma":
        p = c["steps"] + ITERS
        return {"bytes": 2.0 * n * n * p, "flops": 2.0 * n * n * p}
    if kind in ("solve", "refined"):
        p = c["steps"] + ITERS
        return {"bytes": e * ESIZE[c["dtype"]] * p, "flops": 4 * e * p}
    if kind == "frontier":
        return {"bytes": e * ESIZE[c["dtype"]] * (c["steps"] + ITERS), "flops": 4 * e * (c["steps"] + ITERS * c["targets"])}
    if kind == "adjoint":  # 50 products of the estimate; forward, its recomputation and the reverse; the outer products of dL
        p = 50 + 3 * c["iters"]
        return {"bytes": 4 * e * (p + 1), "flops": 4 * e * (p + c["iters"])}
    if kind == "center":
        return {"bytes": e * (4 + ESIZE[c["dtype"]]) + 12.0 * n, "flops": 6 * e}
    if kind == "sigma":
        return {"bytes": e * ESIZE[c["dtype"]] + 4.0 * n * n, "flops": float(n) * (n + 1) * T}
    if kind == "sketch":
        return {"bytes": e * ESIZE[c["dtype"]] + 2.0 * T * c["m"] + 4.0 * n * c["m"], "flops": 2 * e * c["m"]}
    if kind == "countsketch":
        return {"bytes": e * ESIZE[c["dtype"]] + 5.0 * T + 4.0 * n * c["m"], "flops": e}
    n, m, k = c["n"], c["m"], c["k"]  # truncate: the Gram matrix and a few products of it with a block of about 2k columns
    return {"bytes": 4.0 * n * m + 4.0 * n * k, "flops": float(n) * n * m + 20.0 * n * n * k}


# ------------------------------------------------------------------ in 64 bits


def _support(V, mu, nu):
    """Supports of the simplex projections of V + nu mu, for rows V [B, n] and values nu [B, K]: a mask [B, K, n]."""
    W = V[:, None, :] + nu[:, :, None] * mu
    s = W.sort(dim=-1, descending=True).values
    k = torch.arange(1, W.shape[-1] + 1, device=W.device, dtype=F64)
    t = (s.cumsum(-1) - 1) / k
    rho = (s > t).sum(-1, keepdim=True)
    tau = t.gather(-1, rho - 1)
    return W > tau, (W - tau).clamp_min_(0) @ mu


def _search(V, mu, R):
    """Per row of V [B, n]: the support of its projection onto {mu x >= R, 1 x = 1, x >= 0}, and whether the return row is tight."""
    B, K = V.shape[0], 16
    at0, phi0 = _support(V, mu, torch.zeros((B, 1), dtype=F64, device=V.device))
    tight = phi0[:, 0] < R
    lo, hi = torch.zeros(B, dtype=F64, device=V.device), torch.ones(B, dtype=F64, device=V.device)
    while True:
        low = tight & (_support(V, mu, hi[:, None])[1][:, 0] < R)
        if not bool(low.any()):
            break
        lo, hi = torch.where(low, hi, lo), torch.where(low, 4 * hi, hi)
    f = torch.linspace(0, 1, K + 2, dtype=F64, device=V.device)[1:-1]
    for _ in range(9):
        at = lo[:, None] + (hi - lo)[:, None] * f
        under = (_support(V, mu, at)[1] < R[:, None]).sum(1, keepdim=True)
        edges = torch.cat([lo[:, None], at, hi[:, None]], 1)
        lo, hi = edges.gather(1, under)[:, 0], edges.gather(1, under + 1)[:, 0]
    S = _support(V, mu, 0.5 * (lo + hi)[:, None])[0][:, 0]
    return torch.where(tight[:, None], S, at0[:, 0]), tight


def _on_support(V, mu, R, S, tight):
    """The projection whose support is S, from the budget and return rows (differentiable in V and mu)."""
    S = S.to(F64)
    a, b, q = S.sum(-1), S @ mu, S @ (mu * mu)
    sv, smv = (S * V).sum(-1), (S * V) @ mu
    det = torch.where(tight, a * q - b * b, torch.ones_like(a))
    nu = torch.where(tight, (b * (sv - 1) - a * (smv - R)) / det, torch.zeros_like(a))
    tau = (sv + nu * b - 1) / a
    return S * (V + nu[:, None] * mu - tau[:, None])


def _project(V, mu, R):
    return _on_support(V, mu, R, *_search(V, mu, R))


def _estimate(mul, u, steps, lanczos):
    """The largest eigenvalue that `steps` Lanczos or power steps from u see."""
    u = u / u.norm()
    if not lanczos:
        for _ in range(steps):
            u = mul(u)
            u = u / u.norm()
        return float(u @ mul(u))
    a, b, last, beta = [], [], torch.zeros_like(u), 0.0
    for _ in range(steps):
        w = mul(u) - beta * last
        a.append(float(w @ u))
        w = w - a[-1] * u
        beta = float(w.norm())
        b.append(beta)
        last, u = u, w / beta
    return float(np.linalg.eigvalsh(np.diag(a) + np.diag(b[:-1], 1) + np.diag(b[:-1], -1))[-1])


def _npga(mul, gamma, mu, R, alpha, eps, X=None, most=10000):
    """NPGA with a fixed step over rows [B, n] (targets R [B]), each until its own KKT residual, tested every 5, is at most eps: (X, f)."""
    if X is None:
        X = _project(torch.full((R.numel(), mu.numel()), 1.0 / mu.numel(), dtype=F64, device=mu.device), mu, R)
    grad = lambda Z: 2 * mul(Z.T).T + 2 * gamma * Z  # noqa: E731
    Y, t, k = X.clone(), 1.0, 0
    going = torch.ones(R.numel(), dtype=torch.bool, device=mu.device)
    while k < most:
        new = _project(Y - alpha * grad(Y), mu, R)
        s = (1 + math.sqrt(1 + 4 * t * t)) / 2
        beta, t, k = (t - 1) / s, s, k + 1
        Y = new + beta * (new - X)
        X = torch.where(going[:, None], new, X) if not bool(going.all()) else new
        if k % 5 == 0 and eps > 0:
            going &= (_project(X - alpha * grad(X), mu, R) - X).norm(dim=1) > eps
            if not bool(going.any()):
                break
    return X, (X * mul(X.T).T).sum(1) + gamma * X.square().sum(1)


def _solved(L, gamma, mu, R, start, steps, lanczos, explicit=False, then=None):
    """A whole solve on the 64-bit factor (or covariance) L; `then`: the factor that finishes it."""
    mul = (lambda Z: L @ Z) if explicit else (lambda Z: L @ (L.T @ Z))
    alpha = 0.5 / (_estimate(mul, start, steps, lanczos) * (1 + 1e-3) + gamma)
    X, f = _npga(mul, gamma, mu, R, alpha, 1e-5 if then is not None else 1e-6)
    if then is not None:
        X, f = _npga(lambda Z: then @ (then.T @ Z), gamma, mu, R, alpha / 1.01, 1e-6, X)
    return X, f


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind in ("solve", "refined"):
        d = _problem(c, seed)
        R = torch.tensor([d["target"]], dtype=F64, device=DEV)
        n, T, layout = c["n"], c["T"], c["layout"]
        if layout == "sigma":
            L = d["L"][:, :n].to(F64)
            L = torch.triu(L) + torch.triu(L, 1).T
        else:
            L = _wide(d["L"], d["scale"], c["dtype"], "nt" if layout == "str" else layout, n, T)
        then = _wide(d["L_hi"], None, "f32", "tn", n, T) if kind == "refined" else None
        X, f = _solved(L, d["gamma"], d["mu"], R, d["start"], c["steps"], c.get("lanczos", True), layout == "sigma", then)
        return {"x": X[0], "objective": float(f[0]), "iterations": None}
    if kind == "frontier":
        d = _problem(dict(c, layout="nt"), seed)
        L = _wide(d["L"], d["scale"], c["dtype"], "nt", c["n"], c["T"])
        X, f = _solved(L, 0.0, d["mu"], _frontier_targets(d["mu"], c["targets"]), d["start"], c["steps"], True)
        return {"X": X, "objective": f, "iterations": None}
    if kind == "batch":
        xs = []
        for j, (n, T) in enumerate(_batch_sizes(c)):
            if j >= 8:  # the first eight speak for all
                xs.append(None)
                continue
            q = _batch_problem(c, seed, j, n, T)
            X, _ = _solved(_wide(q["L"], None, c["dtype"], c["layout"], n, T), 0.0, q["mu"], torch.tensor([q["R_target"]], dtype=F64, device=DEV),
                           q["power_start"], c["steps"], False)
            xs.append(X[0])
        return {"x": xs, "objective": None, "iterations": None}
    if kind == "adjoint":
        L, mu, target, w = _adjoint_inputs(c, seed)
        n, T, R = c["n"], c["T"], torch.tensor([target], dtype=F64, device=DEV)
        L = L[:, :T].to(F64)
        alpha = 0.5 / (_estimate(lambda u: L @ (L.T @ u), torch.ones(n, dtype=F64, device=DEV), 50, False) * (1 + 1e-3))
        X = _project(torch.full((1, n), 1.0 / n, dtype=F64, device=DEV), mu, R)
        m = mu.clone().requires_grad_()
        Y, t, tape = X, 1.0, []
        for _ in range(c["iters"]):
            Z = Y @ L
            V = Y - 2 * alpha * (Z @ L.T)
            at = _search(V, mu, R)
            s = (1 + math.sqrt(1 + 4 * t * t)) / 2
            new = _on_support(V, mu, R, *at)
            tape.append((Y, Z, V, at, (t - 1) / s))
            X, Y, t = new, new + (t - 1) / s * (new - X), s
        dL, dmu = torch.zeros_like(L), torch.zeros_like(mu)
        gx, gy, gprev = w[None], torch.zeros_like(X), torch.zeros_like(X)
        for Y, Z, V, at, beta in reversed(tape):  # Y_next = (1 + beta) X_next - beta X
            gnew = gx + (1 + beta) * gy
            gprev = -beta * gy
            V = V.requires_grad_()
            gv, gm = torch.autograd.grad(_on_support(V, m, R, *at), (V, m), gnew)
            dmu += gm
            W = gv @ L
            dL.addmm_(gv.T, Z, alpha=-2 * alpha).addmm_(Y.T, W, alpha=-2 * alpha)
            gy = gv - 2 * alpha * (W @ L.T)
            gx = gprev
        return {"x": X[0], "dL": dL, "dmu": dmu}
    if kind == "center":
        mu, L = _centred(_returns(_gen(seed), c["n"], c["T"], 20, 0.01, 0.03))
        trace = L.square().sum().reshape(1)
        if c["dtype"] == "fp8":
            return {"L": None, "mu": mu, "trace": trace, "scale": L.abs().amax(1) / 448}
        L = L.T if c["layout"] == "tn" else L
        return {"L": torch.nn.functional.pad(L, (0, mv.padded_ld(L.shape[1], mv.DTYPES[c["dtype"]]) - L.shape[1])), "mu": mu, "trace": trace}
    if kind == "sigma":
        L, scale, _ = _sketch_inputs(dict(c, m=1), seed)
        L = _wide(L, scale, c["dtype"], "nt", c["n"], c["T"])
        return torch.nn.functional.pad(L @ L.T, (0, -c["n"] % 4))
    if kind == "sketch":
        L, scale, Phi = _sketch_inputs(c, seed)
        return _wide(L, scale, c["dtype"], "nt", c["n"], c["T"]) @ Phi[:, :c["T"]].to(F64).T
    if kind == "countsketch":
        L, scale, (h, sign) = _sketch_inputs(c, seed)
        L = _wide(L, scale, c["dtype"], c["layout"], c["n"], c["T"])
        return torch.zeros((c["n"], c["m"]), dtype=F64, device=DEV).index_add_(1, h.long(), L * sign.to(F64))
    X, trace = _sketched(c, seed)
    X = X.to(F64)
    s2 = torch.linalg.eigvalsh(X @ X.T).flip(0)[:c["k"]]
    return {"L_eff": None, "sigma": s2.sqrt(), "gamma": 1e-4 * trace / c["n"]}

"""The calls that a user of the library makes, over the range of sizes they are made at.

Every case is one pass through the public entry points on a jittered-grid field over
the unit square (the library's synthetic workload), with measurements that are a draw
of the very field whose likelihood is asked for.  `listed` holds the standing cases,
`draw` gives more of the same ranges, `exact` the 64-bit values by plain torch.
"""
import math

import numpy as np
import torch

import paper_1708_02835_gb300 as egs

FEATURES = 1024     # spectral features of the synthetic measurements
QUAD_H = 0.2        # step of the trapezoidal rule for K_nu
QUAD_T = 16.0       # its upper end
EXACT_MAX_N = 26000


def listed():
    return [
        # one likelihood of a small ragged field: what an optimiser on a few hundred stations calls
        {"name": "fp64-777", "kind": "loglik", "precision": "fp64", "n": 777, "tile": 0, "th1": 1.3, "th2": 0.05,
         "nu": 0.8},
        # the small standing workload: 40 x 40 grid, tile 320, exponential model
        {"name": "fp64-1600", "kind": "loglik", "precision": "fp64", "n": 1600, "tile": 320, "th1": 1.0, "th2": 0.1,
         "nu": 0.5},
        # an ordinary FP64 evaluation of a general smoothness (the Bessel path), default tile, ragged
        {"name": "fp64-5000", "kind": "loglik", "precision": "fp64", "n": 5000, "tile": 0, "th1": 1.0, "th2": 0.1,
         "nu": 1.3},
        # a large FP64 evaluation (130 x 130 grid, default tile): the plain exact method at scale
        {"name": "fp64-16900", "kind": "loglik", "precision": "fp64", "n": 16900, "tile": 0, "th1": 1.0, "th2": 0.1,
         "nu": 0.5},
        # one step of a mixed-precision maximum-likelihood fit (160 x 160 grid)
        {"name": "fp32-25600", "kind": "loglik", "precision": "fp32", "n": 25600, "tile": 512, "th1": 1.0,
         "th2": 0.05, "nu": 0.5},
        # the headline size: 320 x 320 grid, mixed precision, resident workspace (a range short enough that
        # the call's accuracy guard passes every draw of the measurements)
        {"name": "fp32-102400", "kind": "loglik", "precision": "fp32", "n": 102400, "tile": 512, "th1": 1.0,
         "th2": 0.03, "nu": 0.5},
        # the TF32 variant on an ordinary rough field, default tile
        {"name": "tf32-10000", "kind": "loglik", "precision": "tf32", "n": 10000, "tile": 0, "th1": 1.2, "th2": 0.04,
         "nu": 0.55},
        # many independent problems of uneven size in one plan (regional fits)
        {"name": "batch-96", "kind": "batch", "count": 96, "n_lo": 256, "n_hi": 4096},
        # kriging of 10,000 new locations from 6,400 observed ones, general smoothness
        {"name": "predict-6400-10000", "kind": "predict", "n": 6400, "m": 10000, "th1": 1.5, "th2": 0.05, "nu": 1.2},
        # the independent-blocks approximation of the headline field (blocks of 1,024)
        {"name": "ind-102400", "kind": "ind", "n": 102400, "tile": 128, "super_tiles": 8, "th1": 1.0, "th2": 0.1,
         "nu": 0.5},
        # Sigma(theta) alone, for a caller with solvers of their own (general smoothness)
        {"name": "matern-25600", "kind": "matern", "n": 25600, "tile": 512, "th1": 1.0, "th2": 0.2, "nu": 1.3},
        # concurrent optimisers: a burst of requests over resident fields, FP64 and mixed
        {"name": "serve-16", "kind": "serve", "requests": 16, "fields": 8, "n_lo": 1000, "n_hi": 8000},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fp64", "fp64", "fp32", "fp32", "tf32", "batch", "predict", "ind", "matern", "serve"])
    th1, nu = round(rng.uniform(0.5, 2.0), 4), rng.choice([0.5, 1.5, round(rng.uniform(0.3, 1.4), 4)])
    th2 = round(rng.uniform(0.03, 0.12), 5)
    if kind == "fp64":
        n = _log_int(rng, 300, 16900)
        tile = rng.choice([0, 0, 128, 256, 320, 512]) if n > 1000 else 0
        return {"kind": "loglik", "precision": "fp64", "n": n, "tile": tile, "th1": th1, "th2": th2, "nu": nu}
    if kind == "fp32":
        n = _log_int(rng, 4000, 102400)
        return {"kind": "loglik", "precision": "fp32", "n": n, "tile": 0 if n < 25000 else 512, "th1": th1,
                "th2": round(rng.uniform(0.015, 0.03), 5), "nu": rng.choice([0.5, 0.5, round(rng.uniform(0.4, 0.5), 4)])}
    if kind == "tf32":
        n = _log_int(rng, 3000, 16000)
        return {"kind": "loglik", "precision": "tf32", "n": n, "tile": 0, "th1": th1,
                "th2": round(rng.uniform(0.02, 0.04), 5), "nu": rng.choice([0.5, round(rng.uniform(0.4, 0.55), 4)])}
    if kind == "batch":
        lo = rng.choice([128, 256, 500])
        return {"kind": "batch", "count": rng.randint(8, 96), "n_lo": lo, "n_hi": lo * rng.randint(2, 8)}
    if kind == "predict":
        return {"kind": "predict", "n": _log_int(rng, 500, 6400), "m": _log_int(rng, 100, 10000), "th1": th1,
                "th2": th2, "nu": nu}
    if kind == "ind":
        return {"kind": "ind", "n": _log_int(rng, 5000, 102400), "tile": rng.choice([0, 64, 128]),
                "super_tiles": rng.randint(1, 8), "th1": th1, "th2": th2, "nu": nu}
    if kind == "matern":
        return {"kind": "matern", "n": _log_int(rng, 1000, 25600), "tile": rng.choice([128, 256, 512]), "th1": th1,
                "th2": th2, "nu": nu}
    return {"kind": "serve", "requests": rng.randint(3, 16), "fields": rng.randint(2, 8), "n_lo": 1000,
            "n_hi": rng.randint(1500, 8000)}


# ---- inputs -----------------------------------------------------------------

def _rng(seed, tag):
    return np.random.default_rng([int(seed) & 0x7FFFFFFF, tag])


def _grid(n, seed, origin=(0.0, 0.0), side=1.0):
    """n locations of a jittered m x m grid, row by row: 2n doubles (x then y) on the GPU."""
    m = math.isqrt(n - 1) + 1
    g = torch.Generator(device="cuda").manual_seed(int(seed) & 0x7FFFFFFF)
    jit = torch.rand(2, n, generator=g, device="cuda", dtype=torch.float64) * 0.8 - 0.4
    i = torch.arange(n, device="cuda")
    rc = torch.stack([i // m, i % m]).to(torch.float64)
    org = torch.tensor(origin, device="cuda", dtype=torch.float64)[:, None]
    return (org + side * (rc + 0.5 + jit) / m).reshape(-1).contiguous()


def _field(locs, n, theta, seed):
    """A zero-mean draw with the Matern covariance by random spectral features: frequencies from its
    spectral density (a bivariate t distribution with 2 nu degrees of freedom), uniform phases."""
    r = _rng(seed, 1)
    th1, th2, nu = theta
    chi2 = 2.0 * r.gamma(nu, size=FEATURES)
    om = r.standard_normal((2, FEATURES)) / (th2 * np.sqrt(chi2))
    ph = r.uniform(0.0, 2.0 * math.pi, FEATURES)
    om, ph = torch.as_tensor(om).cuda(), torch.as_tensor(ph).cuda()
    xy = locs.view(2, n)
    z = torch.empty(n, device="cuda", dtype=torch.float64)
    for a in range(0, n, 16384):
        s = xy[:, a:a + 16384]
        z[a:a + 16384] = torch.cos(s.t() @ om + ph).sum(1)
    return z * math.sqrt(2.0 * th1 / FEATURES)


def _theta(case):
    return (case["th1"], case["th2"], case["nu"])


def _problem(n, theta, seed, origin=(0.0, 0.0), side=1.0):
    locs = _grid(n, seed, origin, side)
    return {"n": n, "theta": theta, "locs": locs, "z": _field(locs, n, theta, seed)}


def _batch_problems(case, seed):
    """Sizes are the case's own; theta, the sub-square and the field of each problem come from the seed."""
    r, sizes = _rng(seed, 2), _rng(case["count"], 4)
    out = []
    for k in range(case["count"]):
        n = int(sizes.integers(case["n_lo"], case["n_hi"] + 1))
        theta = (float(r.uniform(0.5, 2.0)), float(r.uniform(0.03, 0.12)), float(r.uniform(0.3, 1.5)))
        side = float(r.uniform(0.3, 1.0))
        org = tuple(float(v) for v in r.uniform(0.0, 1.0 - side, 2))
        out.append(_problem(n, theta, seed * 1000 + k, org, side))
    return out


def _serve_problems(case, seed):
    """The resident fields and the requests (field, theta, precision); the sizes are the case's own."""
    fields = []
    for k in range(case["fields"]):
        f = k / max(1, case["fields"] - 1)
        n = int(round(math.exp(math.log(case["n_lo"]) * (1 - f) + math.log(case["n_hi"]) * f)))
        fields.append(_problem(n, (1.0, 0.06, 0.5), seed * 100 + k))
    r = _rng(seed, 3)
    reqs = []
    for q in range(case["requests"]):
        theta = (float(r.uniform(0.8, 1.25)), float(r.uniform(0.04, 0.08)), 0.5 if q % 4 else float(r.uniform(0.4, 0.6)))
        reqs.append(((5 * q) % case["fields"], theta, "fp32" if q % 2 else "fp64"))
    return fields, reqs


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        probs = _batch_problems(case, seed)
        return {"kind": kind, "locs": [p["locs"] for p in probs], "z": [p["z"] for p in probs],
                "theta": np.array([p["theta"] for p in probs]), "plan": egs.egs_batch([p["n"] for p in probs])}
    if kind == "serve":
        fields, reqs = _serve_problems(case, seed)
        srv = egs.egs_server(150 * 10 ** 9, max_inflight=8, fallback_fp64=True)
        ids = [srv.add_field(f["locs"], f["z"], f["n"]) for f in fields]
        return {"kind": kind, "server": srv, "requests": [(ids[f], th, p) for f, th, p in reqs]}
    s = _problem(case["n"], _theta(case), seed)
    s["kind"] = kind
    if kind == "loglik":
        p = case["precision"]
        s.update(precision=p, tile=case["tile"], xband=3 if p == "fp32" else 0, workspace=None)
        if case["n"] > 50000:  # a caller at this size keeps the workspace
            s["workspace"] = torch.empty(egs.egs_loglik_workspace_bytes(case["n"], case["tile"], p, 2),
                                         dtype=torch.uint8, device="cuda")
    elif kind == "predict":
        g = torch.Generator(device="cuda").manual_seed((int(seed) + 77) & 0x7FFFFFFF)
        s["new"] = torch.rand(2 * case["m"], generator=g, device="cuda", dtype=torch.float64)
        s["m"] = case["m"]
        s["out"] = torch.empty(case["m"], device="cuda", dtype=torch.float64)
    elif kind == "ind":
        s.update(tile=case["tile"], super_tiles=case["super_tiles"])
    elif kind == "matern":
        s["tile"] = case["tile"]
        s["out"] = torch.empty(egs.egs_tiles_bytes(case["n"], case["tile"]) // 8, device="cuda", dtype=torch.float64)
    return s


def _values(ll, info, precision):
    """l, log|Sigma| and Z' Sigma^-1 Z: doubles from an FP64 evaluation, the numbers the call gives from a mixed one."""
    v = [ll, info["logdet"], info["quad"]]
    return np.array(v) if precision == "fp64" else v


def run(s):
    kind = s["kind"]
    if kind == "loglik":
        kw = {} if s["workspace"] is None else {"workspace": s["workspace"]}
        ll, info = egs.egs_loglik_ex(s["locs"], s["z"], s["theta"], s["n"], s["precision"], tile=s["tile"],
                                     xband=s["xband"], **kw)
        return _values(ll, info, s["precision"])
    if kind == "batch":
        out, stat = s["plan"].run(s["locs"], s["z"], s["theta"])
        return [out, stat]
    if kind == "predict":
        info = egs.egs_predict(s["locs"], s["z"], s["n"], s["new"], s["m"], s["theta"], s["out"])
        return [s["out"], _values(info["loglik"], info, "fp64")]
    if kind == "ind":
        ll, info = egs.egs_loglik_ind(s["locs"], s["z"], s["theta"], s["n"], tile=s["tile"],
                                      super_tiles=s["super_tiles"])
        return _values(ll, info, "fp64")
    if kind == "matern":
        egs.egs_matern_tiles(s["locs"], s["n"], s["theta"], s["tile"], s["out"])
        return s["out"]
    srv = s["server"]
    tickets = [srv.submit(f, th, p) for f, th, p in s["requests"]]
    got = [srv.wait(t)[0] for t in tickets]
    return [np.array([v for v, r in zip(got, s["requests"]) if r[2] == "fp64"]),
            [v for v, r in zip(got, s["requests"]) if r[2] != "fp64"]]


# ---- work -------------------------------------------------------------------

def _loglik_work(n):
    """Locations and measurements in; n^2 / 2 covariances (about 20 operations each), the Cholesky, the solve."""
    return {"bytes": 24.0 * n + 24.0, "flops": n ** 3 / 3.0 + 10.0 * n * n + n * n}


def work(case):
    kind = case["kind"]
    if kind == "loglik":
        return _loglik_work(case["n"])
    if kind == "predict":
        w = _loglik_work(case["n"])
        return {"bytes": w["bytes"] + 24.0 * case["m"], "flops": w["flops"] + 22.0 * case["n"] * case["m"]}
    if kind == "ind":
        bs = (case["tile"] or 128) * case["super_tiles"]
        ns = [min(bs, case["n"] - a) for a in range(0, case["n"], bs)]
    elif kind == "matern":
        t = -(-case["n"] // case["tile"])
        return {"bytes": 16.0 * case["n"] + 4.0 * t * (t + 1) * case["tile"] ** 2, "flops": 10.0 * case["n"] ** 2}
    elif kind == "batch":
        sizes = _rng(case["count"], 4)
        ns = [int(sizes.integers(case["n_lo"], case["n_hi"] + 1)) for _ in range(case["count"])]
    else:
        ns, f = [], case["fields"]
        for q in range(case["requests"]):
            w = ((5 * q) % f) / max(1, f - 1)
            ns.append(math.exp(math.log(case["n_lo"]) * (1 - w) + math.log(case["n_hi"]) * w))
    ws = [_loglik_work(n) for n in ns]
    return {"bytes": sum(w["bytes"] for w in ws), "flops": sum(w["flops"] for w in ws)}


# ---- 64-bit values ----------------------------------------------------------

def _cov(r, theta):
    """The Matern covariance of a tensor of distances: closed forms at nu = 1/2 and 3/2, else K_nu by the
    trapezoidal rule on its integral over exp(-x cosh t) cosh(nu t)."""
    th1, th2, nu = theta
    x = r / th2
    if nu == 0.5:
        return th1 * torch.exp(-x)
    if nu == 1.5:
        return th1 * (1.0 + x) * torch.exp(-x)
    acc = torch.exp(-x) * (0.5 * QUAD_H)
    t = QUAD_H
    while t <= QUAD_T:
        acc += torch.exp(x * -math.cosh(t)) * (QUAD_H * math.cosh(nu * t))
        t += QUAD_H
    c = acc * x ** nu * (th1 / (2.0 ** (nu - 1.0) * math.gamma(nu)))
    return torch.where(x > 0.0, c, torch.full_like(c, th1))


def _cross(a, b, theta, out=None):
    """Covariances of locations a (2, p) with b (2, q), some rows at a time."""
    out = torch.empty(a.shape[1], b.shape[1], device="cuda", dtype=torch.float64) if out is None else out
    step = max(1, 2 ** 25 // b.shape[1])
    for i in range(0, a.shape[1], step):
        d = a[:, i:i + step, None] - b[:, None, :]
        out[i:i + step] = _cov(torch.hypot(d[0], d[1]), theta)
    return out


def _loglik_exact(locs, z, n, theta, solve=False):
    xy = locs.view(2, n)
    chol = torch.linalg.cholesky(_cross(xy, xy, theta))
    y = torch.linalg.solve_triangular(chol, z[:, None], upper=False)
    ld, q = 2.0 * float(torch.log(torch.diagonal(chol)).sum()), float((y * y).sum())
    v = [-0.5 * (q + ld + n * math.log(2.0 * math.pi)), ld, q]
    return (v, torch.linalg.solve_triangular(chol.t(), y, upper=True)[:, 0]) if solve else v


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        probs = _batch_problems(case, seed)
        return [np.array([_loglik_exact(p["locs"], p["z"], p["n"], p["theta"])[0] for p in probs]), None]
    if kind == "serve":
        fields, reqs = _serve_problems(case, seed)
        got = [_loglik_exact(fields[f]["locs"], fields[f]["z"], fields[f]["n"], th)[0] for f, th, _ in reqs]
        return [np.array([v for v, r in zip(got, reqs) if r[2] == "fp64"]),
                [np.float64(v) for v, r in zip(got, reqs) if r[2] != "fp64"]]
    n, theta = case["n"], _theta(case)
    p = _problem(n, theta, seed)
    if kind == "ind":
        bs = (case["tile"] or 128) * case["super_tiles"]
        xy, tot = p["locs"].view(2, n), np.zeros(3)
        for a in range(0, n, bs):
            loc = xy[:, a:a + bs].contiguous().reshape(-1)
            tot += np.array(_loglik_exact(loc, p["z"][a:a + bs], min(bs, n - a), theta))
        return tot
    if kind == "matern":
        b = case["tile"]
        t, xy = -(-n // b), p["locs"].view(2, n)
        out = torch.zeros(t * (t + 1) // 2, b, b, device="cuda", dtype=torch.float64)
        k = 0
        for i in range(t):
            a = xy[:, i * b:(i + 1) * b]
            for j in range(i + 1):
                c = xy[:, j * b:(j + 1) * b]
                out[k, :a.shape[1], :c.shape[1]] = _cross(a, c, theta)
                k += 1
        out[-1].diagonal()[n - (t - 1) * b:] = 1.0
        return out.reshape(-1)
    if n > EXACT_MAX_N:
        return None
    if kind == "predict":
        s = prepare(case, seed)
        v, x = _loglik_exact(p["locs"], p["z"], n, theta, solve=True)
        xy, new = p["locs"].view(2, n), s["new"].view(2, case["m"])
        return [_cross(new, xy, theta) @ x, np.array(v)]
    v = _loglik_exact(p["locs"], p["z"], n, theta)
    return np.array(v) if case["precision"] == "fp64" else [np.float64(x) for x in v]

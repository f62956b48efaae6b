"""Workloads for measuring the library: what a program that uses it runs, through the public entry points.

A case names a point cloud, a kernel, the plan's options and one call on the plan: a matvec (the product
inside conjugate gradients and stochastic trace estimates), a conjugate gradient solve capped at a number of
iterations (the usual budget of a hyperparameter search), or a posterior mean at new points.  ``prepare``
builds what such a program holds before the call (the plan, the vectors), ``run`` makes the call.

The point clouds and fields follow ``gpinputs`` (drawn on the GPU here, from the seed).  Results of an FP32
plan are kept in float32, the accuracy such a plan computes to; those of float64 and float-float plans in
float64, as the library returns them.
"""
import math

import torch

import paper_2407_03608_gb300 as gpn

_PRECISION = {"fp32": gpn.GP_FP32, "fp64": gpn.GP_FP64, "df64": gpn.GP_DF64}
_ETA2 = {1: 0.01, 2: 0.0025, 3: 0.01}
_MAX_PAIRS = 1.3e10      # kernel entries that exact() forms within its time
_DENSE_N = 20000         # points up to which exact() keeps the dense matrix (capped solves)


def _case(name, call, d, n, precision, nu, eps, points, fields, rhs=1, block=0, step3=0, iters=0, queries=0):
    c = dict(call=call, d=d, n=n, precision=precision, nu=nu, eps=eps, points=points, fields=fields, rhs=rhs,
             block=block, step3=step3, iters=iters, queries=queries)
    return dict(c, name=name) if name else c


def listed():
    return [
        # 1-D, the smallest workload in daily use: one product, then the solve it sits in (both bound by
        # latency: a dozen short transforms in float64)
        _case("d1-matvec-fp64", "matvec", 1, 2000, "fp64", 1.5, 1e-6, "uniform", "fixed"),
        _case("d1-solve-fp64", "solve", 1, 2000, "fp64", 1.5, 1e-6, "uniform", "fixed", iters=12),
        # a longer series with short length scales and a few right-hand sides, as a solve server gets it
        _case("d1-matvec-fp32-r4", "matvec", 1, 100003, "fp32", 1.5, 1e-6, "uniform", "narrow", rhs=4),
        # a small 2-D request of the server: the grid is small and the launches count
        _case("d2-matvec-fp32-small", "matvec", 2, 5000, "fp32", 2.5, 1e-6, "uniform", "narrow", rhs=3),
        # the 2-D benchmark points in the three arithmetics: the FP32 product of the mixed-precision solve,
        # a few iterations of the float64-grade solve, and a coarser float64 product
        _case("d2-matvec-fp32", "matvec", 2, 1000000, "fp32", 1.5, 1e-6, "clustered", "fixed"),
        _case("d2-solve-df64", "solve", 2, 1000000, "df64", 1.5, 1e-6, "clustered", "fixed", iters=3),
        _case("d2-matvec-fp64", "matvec", 2, 100000, "fp64", 1.5, 1e-4, "clustered", "fixed"),
        # many probe vectors through grids held for a block of them
        _case("d2-probes-fp32", "matvec", 2, 100000, "fp32", 1.5, 1e-5, "clustered", "fixed", rhs=16, block=8),
        # prediction at as many new points as there are training points
        _case("d2-mean-fp32", "mean", 2, 100000, "fp32", 1.5, 1e-5, "clustered", "fixed", queries=100000),
        # 3-D: a large cloud in FP32, a small one in float64, and the largest plan (1e-6 at N = 2e6) with the
        # memory-lean step 3
        _case("d3-matvec-fp32", "matvec", 3, 2000000, "fp32", 2.5, 1e-5, "uniform", "fixed"),
        _case("d3-matvec-fp64", "matvec", 3, 20000, "fp64", 2.5, 1e-4, "uniform", "fixed"),
        _case("d3-matvec-fp32-lean", "matvec", 3, 2000000, "fp32", 2.5, 1e-6, "uniform", "fixed", step3=2),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the same ranges: sizes spread over their logarithm, options as they occur together."""
    d = rng.choice((1, 1, 2, 2, 2, 3, 3))
    call = rng.choice(("matvec", "matvec", "matvec", "solve", "mean"))
    fields = rng.choice(("fixed", "narrow"))
    points = "clustered" if d == 2 and rng.random() < 0.5 else "uniform"
    precision = rng.choice(("fp32", "fp32", "fp64") if d != 2 else ("fp32", "fp32", "fp64", "df64"))
    nu = rng.choice((1.5, 2.5)) if d < 3 else 2.5
    if d == 1:
        eps = rng.choice((1e-4, 1e-5, 1e-6))
        if rng.random() < 0.2:
            nu, eps = 0.5, 1e-2
        n, rhs = _log_uniform(rng, 1000, 1000000), rng.choice((1, 1, 2, 5, 16))
    elif d == 2:
        eps = rng.choice((1e-3, 1e-4, 1e-5)) if precision != "fp64" else rng.choice((1e-3, 1e-4))
        n, rhs = _log_uniform(rng, 1000, 1000000), rng.choice((1, 1, 2, 5, 16))
    else:
        eps = rng.choice((1e-3, 1e-4)) if precision == "fp64" else rng.choice((1e-3, 1e-4, 1e-5))
        n, rhs = _log_uniform(rng, 1000, 2000000 if precision == "fp32" else 200000), rng.choice((1, 1, 2))
        fields = "fixed"
    block = rng.choice((0, 0, 2, 4)) if rhs > 2 else 0
    if d == 2 and rhs == 16:
        block = 4
    step3 = 2 if precision == "fp32" and d > 1 and rng.random() < 0.2 else 0
    iters, queries = 0, 0
    if call == "solve":
        iters = rng.randint(2, 6)
        precision = "fp64" if d != 2 else rng.choice(("fp64", "df64"))
        rhs, block, step3 = rng.choice((1, 2)), 0, 0
        n = min(n, 200000)
        eps = max(eps, 1e-4) if d > 1 else eps
    elif call == "mean":
        rhs, block = 1, 0
        queries = _log_uniform(rng, 100, 200000)
    return _case(None, call, d, n, precision, nu, eps, points, fields, rhs, block, step3, iters, queries)


# ---- inputs ---------------------------------------------------------------------------------------------

def _points(g, n, d, kind):
    if kind == "uniform":
        return torch.rand((n, d), generator=g, device="cuda", dtype=torch.float64)
    half = n // 2
    uni = torch.rand((half, 2), generator=g, device="cuda", dtype=torch.float64)
    centres = 0.1 + 0.8 * torch.rand((8, 2), generator=g, device="cuda", dtype=torch.float64)
    which = torch.arange(n - half, device="cuda") % 8
    noise = torch.randn((n - half, 2), generator=g, device="cuda", dtype=torch.float64)
    # three standard deviations at most, so that every seed's cloud has the same extent
    return torch.cat([uni, centres[which] + 0.03 * noise.clamp(-3.0, 3.0)])


def _fields(x, n, kind):
    """(s, l) at the points x; n, the size of the training set, sets the narrow length scale."""
    d, tau = x.shape[1], 2.0 * math.pi
    if kind == "narrow":   # lengths shrink with the spacing of the points, down to a floor
        l0 = max(0.08 * (n / 1000.0) ** (-1.0 / d), {1: 0.004, 2: 0.02, 3: 0.05}[d])
        wave = torch.cos(tau * x).prod(dim=1)
        return 1.0 + 0.3 * torch.sin(tau * x[:, 0]), l0 * (1.0 + 0.4 * wave)
    if d == 1:
        return 1.0 + 0.5 * torch.sin(tau * x[:, 0]), 0.05 + 0.03 * torch.cos(tau * x[:, 0])
    if d == 2:
        a, b = x[:, 0], x[:, 1]
        return 1.0 + 0.3 * a, 0.02 + 0.02 * (1.0 + torch.sin(tau * a) * torch.cos(tau * b)) / 2.0
    return torch.exp(-((x - 0.5) ** 2).sum(dim=1)), 0.05 + 0.05 * (x ** 2).sum(dim=1) / 3.0


def _inputs(case, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed) * 1000003 + 17)
    n, d = case["n"], case["d"]
    x = _points(g, n, d, case["points"])
    s, l = _fields(x, n, case["fields"])
    if case["call"] == "solve":
        base = torch.sin(12.0 * x[:, 0]) * torch.cos(4.0 * math.pi * x[:, -1])
        noise = torch.randn((case["rhs"], n), generator=g, device="cuda", dtype=torch.float64)
        vec = base + math.sqrt(_ETA2[d]) * noise
    elif case["rhs"] > 1:   # probe vectors
        vec = torch.randint(0, 2, (case["rhs"], n), generator=g, device="cuda").to(torch.float64) * 2.0 - 1.0
    else:
        vec = torch.randn((1, n), generator=g, device="cuda", dtype=torch.float64)
    out = {"x": x, "s": s, "l": l, "vec": vec[0] if case["rhs"] == 1 else vec.t()}
    if case["call"] == "mean":
        # queries inside the cloud: between two training points each
        i = torch.randint(0, n, (case["queries"],), generator=g, device="cuda")
        t = torch.rand((case["queries"], 1), generator=g, device="cuda", dtype=torch.float64)
        q = x[i] * t + x[i.flip(0)] * (1.0 - t)
        sq, lq = _fields(q, n, case["fields"])
        out.update(q=q, sq=sq, lq=lq.clamp(float(l.min()), float(l.max())))
    return out


def prepare(case, seed):
    data = _inputs(case, seed)
    opts = {"step3": case["step3"]} if case["step3"] else {}
    if case["block"]:
        opts["rhs_block"] = case["block"]
    plan = gpn.Plan(data["x"], data["s"], data["l"], nu=case["nu"], eps=case["eps"],
                    precision=_PRECISION[case["precision"]], max_rhs=case["rhs"], **opts)
    return {"case": case, "plan": plan, "data": data}


def run(state):
    case, plan, data = state["case"], state["plan"], state["data"]
    if case["call"] == "matvec":
        out = plan.matvec(data["vec"], shift=_ETA2[case["d"]])
    elif case["call"] == "solve":
        out, _ = plan.solve(data["vec"], eta2=_ETA2[case["d"]], rtol=1e-12, maxit=case["iters"])
    else:
        out = plan.posterior_mean(data["vec"], data["q"], data["sq"], data["lq"])
    return out.to(torch.float32) if case["precision"] == "fp32" else out


# ---- what a pass cannot do without ----------------------------------------------------------------------

def work(case):
    """Bytes: the call's vectors, the per-point data (coordinates and the two fields), and step 3's tensor or
    factors.  Operations: spreading and interpolation (a multiply-add per point, channel and support cell),
    the transforms of the occupied part of the grid, step 3."""
    o = gpn.abi.default_opts(precision=_PRECISION[case["precision"]], max_rhs=case["rhs"], step3=case["step3"])
    n, d, r = case["n"], case["d"], case["rhs"]
    floor = {1: 0.004, 2: 0.02, 3: 0.05}[d]
    if case["fields"] == "narrow":
        l0 = max(0.08 * (n / 1000.0) ** (-1.0 / d), floor)
        lo, hi = 0.6 * l0, 1.4 * l0
    else:
        lo, hi = {1: (0.02, 0.08), 2: (0.02, 0.04), 3: (0.05, 0.10)}[d]
    i = gpn.abi.gp_plan_params(d, n, case["nu"], case["eps"], lo, hi, [0.0] * d, [1.0] * d, o)
    c, w, modes = i["n_sigma"] + 1, i["kernel_width"], 2 * i["M"] + 1
    size = 4 if case["precision"] == "fp32" else 8
    freqs = modes ** (d - 1) * (i["M"] + 1)
    tensor = c * (c + 1) // 2 * (i["M"] + 1) * (i["M"] + 1 if d == 2 else modes ** (d - 1)) * size
    lean = c * (i["n_t"] + 1) * (i["M"] + 1) * size
    passes = max(1, case["iters"])
    points = 8.0 * n * (d + 2) + 8.0 * case["queries"] * (d + 3)
    once = (lean if case["step3"] == 2 else tensor) + points + 16.0 * n * r
    occupied = (i["dw"] * i["nf"]) * i["nf"] ** (d - 1) * i["dw"] ** (d - 1)
    fft = 2.0 * 2.5 * c * r * d * max(occupied, float(freqs)) * math.log2(i["nf"])
    spread = 2.0 * r * c * w ** d * (n + (case["queries"] or n))
    step3 = freqs * r * c * (16.0 * (i["n_t"] + 1) if case["step3"] == 2 else 4.0 * c)
    return {"bytes": once * passes, "flops": (fft + spread + step3) * passes}


# ---- the same in 64 bits --------------------------------------------------------------------------------

def _phi(r, nu):
    if nu == 0.5:
        return torch.exp(-r)
    a = r * math.sqrt(2.0 * nu)
    poly = 1.0 + a if nu == 1.5 else 1.0 + a + a * a / 3.0
    return poly * torch.exp(-a)


def _block(x, s, l, y, sy, ly, nu):
    """K(x_i, y_j) = s_i s_j (l_i l_j)^(d/2) / m_ij^(d/2) phi_nu(|x_i - y_j| / sqrt(m_ij)), m = (l_i^2 + l_j^2) / 2."""
    d = x.shape[1]
    m = 0.5 * (l[:, None] ** 2 + ly[None, :] ** 2)
    r2 = torch.zeros_like(m)
    for a in range(d):
        r2 += (x[:, a, None] - y[None, :, a]) ** 2
    k = _phi(torch.sqrt(r2 / m), nu)
    k *= torch.sqrt(l[:, None] * ly[None, :] / m) ** d
    return k * (s[:, None] * sy[None, :])


def _apply(x, s, l, y, sy, ly, nu, v):
    rows = max(1, int(1.5e8 // y.shape[0]))
    return torch.cat([_block(x[i:i + rows], s[i:i + rows], l[i:i + rows], y, sy, ly, nu) @ v
                      for i in range(0, x.shape[0], rows)])


def exact(case, seed):
    n = case["n"]
    if float(n) * (case["queries"] or n) > _MAX_PAIRS or (case["call"] == "solve" and n > _DENSE_N):
        return None
    t, nu, eta2 = _inputs(case, seed), case["nu"], _ETA2[case["d"]]
    x, s, l, v = t["x"], t["s"], t["l"], t["vec"]
    one = v.dim() == 1
    v = v[:, None] if one else v
    if case["call"] == "mean":
        out = _apply(t["q"], t["sq"], t["lq"], x, s, l, nu, v)
    elif case["call"] == "matvec":
        out = _apply(x, s, l, x, s, l, nu, v) + eta2 * v
    else:
        k = _block(x, s, l, x, s, l, nu)
        out, res = torch.zeros_like(v), v.clone()
        p, rr = res.clone(), (res * res).sum(dim=0)
        for _ in range(case["iters"]):
            kp = k @ p + eta2 * p
            a = rr / (p * kp).sum(dim=0)
            out, res = out + a * p, res - a * kp
            new = (res * res).sum(dim=0)
            p, rr = res + (new / rr) * p, new
    return out[:, 0] if one else out

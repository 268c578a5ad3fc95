"""The measured cases: what a user of the library has it do, over its real range of sizes.

Geometry: star-shaped islands on the sphere (radius r0 (1 + a cos k t) about a centre),
the family the benchmark uses (r0 ~ U[0.2, 1] / sqrt(M), a ~ U[0, 0.3], k ~ 2..8), with
centres on a Fibonacci lattice so that any number of islands is placed without a search.
Data: a +1 / -1 pair of point sources inside islands (the exact solution is then the pair's
potential) or, for single operator applications, normal random densities, as a Krylov
vector is.

Kinds of case:
  apply     one operator application on a kept plan (lbf_apply): the step inside GMRES
  solve     one GMRES solve and an evaluation on a kept plan
  many      several right-hand sides of one geometry in lockstep on a kept plan
  evaluate  the potential of a known density at many targets
  gradient  autograd: plan, solve, evaluation and the adjoint solve from planar nodes
  step      the whole call on a new geometry: plan, solve, evaluation
  batch     lbf_batch_run over several uneven geometries
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1306_0612_gb300 import lbfmm as L
from paper_1306_0612_gb300.autograd import solve_evaluate

TWO_PI = 2.0 * math.pi
F64 = torch.float64
OPS = {"full": L.LBF_OP_FULL, "prec": L.LBF_OP_PRECONDITIONED, "density": L.LBF_OP_K_ONLY}


def _dev():
    return torch.device("cuda", torch.cuda.current_device())


# ---- the cases ----------------------------------------------------------------------


def _case(name, kind, M, lo, hi, **kw):
    """M islands of lo..hi nodes (the same number for all where lo = hi).  fmm64: the
    accurate operator's arithmetic, 1 double-float (the library's default) or 0 native
    double (the benchmark's)."""
    c = dict(kind=kind, M=M, lo=lo, hi=hi, p=26, leaf=48, tol=1e-12, fmm64=1)
    c.update(kw)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # one island, 256 nodes, direct sums: the smallest solve (interactive use, latency)
        _case("solve-single-direct", "solve", 1, 256, 256, direct=True, targets=256),
        # one application at the benchmark's small configuration: launches and chains count
        _case("apply-16x512", "apply", 16, 512, 512, op="full"),
        # one application with uneven odd island sizes, the paper's Example 3 island count
        _case("apply-407-ragged", "apply", 407, 131, 1021, op="prec"),
        # the operator inside GMRES at the benchmark's default size (16.8 million nodes)
        _case("apply-16384x1024", "apply", 16384, 1024, 1024, op="prec", p=22, fmm64=0),
        # the adjoint's operator on the gradient workload's shape
        _case("transpose-256x512", "apply", 256, 512, 512, op="full", transpose=True),
        # a solve at the paper's Example 3 size, its tolerance, its number of targets
        _case("solve-407x1024", "solve", 407, 1024, 1024, tol=1e-11, targets=77, fmm64=0),
        # one FP32 refinement solve at a middle size
        _case("solve-refine-1024x512", "solve", 1024, 512, 512, tol=1e-11, refine=True, targets=256),
        # sixteen right-hand sides of one small uneven geometry: the batched workload's unit
        _case("many-24x16rhs", "many", 24, 64, 1021, nrhs=16, fmm64=0),
        # twelve uneven geometries with 16 right-hand sides each, FP32 refinement, whole call
        _case("batch-12", "batch", 64, 64, 511, nrhs=16, count=12, refine=True, inner_tol=1e-5,
              targets=16, fmm64=0),
        # a map of the solution: many targets
        _case("evaluate-128x512", "evaluate", 128, 512, 512, targets=40000),
        # gradient of a loss in the data and the node positions, plan included
        _case("gradient-256x512", "gradient", 256, 512, 512, tol=1e-11, targets=4096, fmm64=0),
        # a new geometry solved from scratch, large enough for the factored preconditioner
        _case("step-2048x1024", "step", 2048, 1024, 1024, p=22, tol=1e-11, targets=256,
              fmm64=0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "solve", "solve", "many", "batch", "evaluate",
                       "gradient", "step"])
    p, leaf = rng.choice([22, 24, 26, 26, 30]), rng.choice([32, 48, 48, 64])
    fmm64 = rng.choice([0, 1])
    lo = _log(rng, 48, 500)
    hi = max(lo, _log(rng, 200, 1100))
    if kind == "apply":
        op = rng.choice(["full", "prec", "density"])
        return _case(None, kind, _log(rng, 2, 4000), lo, hi, op=op, p=p, leaf=leaf,
                     transpose=rng.random() < 0.25, fmm64=fmm64)
    if kind == "solve":
        return _case(None, kind, _log(rng, 2, 700), lo, hi, tol=1e-11, p=max(p, 24), leaf=leaf,
                     refine=rng.random() < 0.4, targets=_log(rng, 16, 1000), fmm64=fmm64)
    if kind == "many":
        return _case(None, kind, _log(rng, 2, 64), min(lo, 200), min(hi, 600), nrhs=rng.randint(2, 16),
                     leaf=leaf, refine=rng.random() < 0.5, fmm64=fmm64)
    if kind == "batch":
        return _case(None, kind, _log(rng, 8, 64), min(lo, 128), min(hi, 512), nrhs=rng.randint(1, 16),
                     count=rng.randint(2, 12), refine=rng.random() < 0.5, targets=16, fmm64=fmm64)
    if kind == "evaluate":
        return _case(None, kind, _log(rng, 1, 400), lo, hi, targets=_log(rng, 500, 50000), fmm64=fmm64)
    if kind == "gradient":
        return _case(None, kind, _log(rng, 2, 256), min(lo, 300), min(hi, 700), tol=1e-11, leaf=leaf,
                     targets=_log(rng, 100, 4000), fmm64=fmm64)
    return _case(None, kind, _log(rng, 8, 1500), lo, hi, tol=1e-11, p=max(p, 24), leaf=leaf,
                 targets=_log(rng, 64, 512), fmm64=fmm64)


# ---- geometry -----------------------------------------------------------------------


class _Geometry:
    """Islands as torch tensors on the GPU (nodes n x 3), host CSR offsets."""


def _geometry(M, lo, hi, rng):
    i = np.arange(M) + 0.5
    z = 1.0 - 2.0 * i / M
    ph = math.pi * (3.0 - math.sqrt(5.0)) * i + rng.uniform(0, TWO_PI)
    s = np.sqrt(1.0 - z * z)
    c = np.stack([s * np.cos(ph), s * np.sin(ph), z], 1)
    c = c[rng.permutation(M)]
    e1, e2 = _frames(c[:1])  # the first centre becomes the north pole
    R = np.concatenate([e1, e2, c[:1]])
    c = c @ R.T
    c[0] = (0.0, 0.0, 1.0)
    e1, e2 = _frames(c)
    scale = min(1.0, math.sqrt(16.0 / M))
    r0 = rng.uniform(0.05, 0.25, M) * scale
    amp = rng.uniform(0.0, 0.3, M)
    kf = rng.integers(2, 9, M).astype(np.float64)
    # the islands' node counts belong to the case, their shapes to the seed
    sizes = np.random.default_rng([M, lo, hi])
    n = np.round(np.exp(sizes.uniform(math.log(lo), math.log(hi), M))).astype(np.int64)
    g = _Geometry()
    g.M, g.ptr = M, np.concatenate([[0], np.cumsum(n)]).astype(np.int64)
    g.N = int(g.ptr[-1])
    g.rmin, g.rmax = r0 * (1 - amp), r0 * (1 + amp)
    g.c_host, g.e1_host = c, e1
    d = _dev()
    up = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(d)  # noqa: E731
    g.c = up(c)
    nt = up(n)
    g.isl = torch.repeat_interleave(torch.arange(M, device=d), nt)
    g.h = (TWO_PI / nt.to(F64))[g.isl]
    t = (torch.arange(g.N, device=d) - up(g.ptr[:-1])[g.isl]).to(F64) * g.h
    r0, amp, kf = up(r0)[g.isl], up(amp)[g.isl], up(kf)[g.isl]
    r = r0 * (1 + amp * torch.cos(kf * t))
    rp = -r0 * amp * kf * torch.sin(kf * t)
    rpp = -r0 * amp * kf * kf * torch.cos(kf * t)
    C, E1, E2 = g.c[g.isl], up(e1)[g.isl], up(e2)[g.isl]
    ct, st = torch.cos(t)[:, None], torch.sin(t)[:, None]
    u, v = ct * E1 + st * E2, ct * E2 - st * E1
    cr, sr = torch.cos(r)[:, None], torch.sin(r)[:, None]
    rp, rpp = rp[:, None], rpp[:, None]
    g.x = cr * C + sr * u
    g.dx = -rp * sr * C + rp * cr * u + sr * v
    g.d2x = (-rpp * sr - rp * rp * cr) * C + (rpp * cr - rp * rp * sr - sr) * u + 2 * rp * cr * v
    return g


def _frames(c):
    ref = np.where(np.abs(c[:, 2:3]) <= 0.9, [[0.0, 0.0, 1.0]], [[1.0, 0.0, 0.0]])
    e1 = np.cross(ref, c)
    e1 /= np.linalg.norm(e1, axis=1, keepdims=True)
    return e1, np.cross(c, e1)


def _planar(g):
    """xi, xi', xi'' (N x 2): the stereographic projection (x1 + i x2)/(1 - x3), chain rule."""
    X, X1, X2 = (torch.complex(a[:, 0].contiguous(), a[:, 1].contiguous()) for a in (g.x, g.dx, g.d2x))
    s, z1, z2 = 1 - g.x[:, 2], g.dx[:, 2], g.d2x[:, 2]
    a = X / s
    b = X1 / s + X * z1 / s**2
    c = X2 / s + 2 * X1 * z1 / s**2 + X * z2 / s**2 + 2 * X * z1**2 / s**3
    return tuple(torch.view_as_real(v).contiguous() for v in (a, b, c))


def _targets(g, T, rng):
    """T points on the sphere outside every island's circumscribed cap."""
    d, got, have = _dev(), [], 0
    lim = torch.from_numpy(np.cos(1.1 * g.rmax)).to(d)
    while have < T:
        n = max(64, min(2 * (T - have) + 64, (1 << 27) // g.M))
        t = rng.standard_normal((n, 3))
        t = torch.from_numpy(t / np.linalg.norm(t, axis=1, keepdims=True)).to(d)
        t = t[(t @ g.c.T < lim).all(dim=1)]
        got.append(t)
        have += len(t)
    return torch.cat(got)[:T].contiguous()


def _sources(g, rng):
    """A +1 / -1 pair of point sources inside two random islands (one where M = 1)."""
    k = (0, 0) if g.M == 1 else tuple(int(v) for v in rng.choice(g.M, 2, replace=False))
    at = [rng.uniform(0.0, 0.3), rng.uniform(0.4, 0.7)]
    pts = [math.cos(f * g.rmin[j]) * g.c_host[j] + math.sin(f * g.rmin[j]) * g.e1_host[j]
           for j, f in zip(k, at)]
    return torch.from_numpy(np.stack(pts)).to(_dev())


def _pair_potential(x, src):
    """G(x, p) - G(x, q): the exact solution of the pair's data."""
    d = [((x - s) ** 2).sum(1) for s in src]
    return (torch.log(d[1]) - torch.log(d[0])) / (2 * TWO_PI)


# ---- what is measured ---------------------------------------------------------------


def _options(c):
    o = L.lbf_default_options(tol=c["tol"], p=c["p"], leaf_size=c["leaf"], fmm64=c["fmm64"])
    if c.get("direct"):
        o.matvec = L.LBF_MATVEC_DIRECT
    if c.get("refine"):
        o.precision = L.LBF_PRECISION_FP32_REFINE
    if c.get("inner_tol"):
        o.inner_tol = c["inner_tol"]
    return o


def _empty(*n):
    return torch.empty(n, dtype=F64, device=_dev())


class _State:
    pass


def _inputs(c, seed):
    """(geometry, the rest of the inputs by name), from the seed alone."""
    rng = np.random.default_rng([seed, 20130602])
    g = _geometry(c["M"], c["lo"], c["hi"], rng)
    gen = torch.Generator(device=_dev())
    gen.manual_seed(seed)
    more = {}
    if c["kind"] in ("apply", "evaluate"):
        more["vec"] = torch.randn(g.N + g.M, dtype=F64, device=_dev(), generator=gen)
        if c["kind"] == "evaluate":
            more["vec"][g.N:] -= more["vec"][g.N:].mean()
    elif c["kind"] in ("many", "batch"):
        more["src"] = [_sources(g, rng) for _ in range(c["nrhs"])]
        more["data"] = torch.stack([_pair_potential(g.x, s) for s in more["src"]])
    else:
        more["src"] = _sources(g, rng)
        more["data"] = _pair_potential(g.x, more["src"])
    if c.get("targets"):
        more["targets"] = _targets(g, c["targets"], rng)
    return g, more


def _plan(g, o):
    return L.lbf_plan_create(g.ptr, g.x, g.dx, g.d2x, g.c, opt=o)


def _many_geometries(c):
    """The batch's geometries: uneven island counts, M / 4 to M."""
    for q in range(c["count"]):
        yield dict(c, M=max(1, round(c["M"] * (0.25 + 0.75 * ((q * 5) % c["count"]) / c["count"]))))


def prepare(case, seed):
    c, s = case, _State()
    s.case, s.opt, kind = c, _options(c), c["kind"]
    if kind == "batch":
        s.items = []
        for q, cq in enumerate(_many_geometries(c)):
            g, m = _inputs(cq, seed * 1000 + q)
            s.items.append(dict(island_ptr=g.ptr, x=g.x, dx=g.dx, d2x=g.d2x, centres=g.c,
                                g=m["data"], targets=m["targets"]))
        return s
    g, m = _inputs(c, seed)
    s.N, s.M, s.ptr = g.N, g.M, g.ptr
    s.targets, s.data, s.vec = m.get("targets"), m.get("data"), m.get("vec")
    if kind == "gradient":
        s.xi, s.dxi, s.d2xi = _planar(g)
        s.c = g.c
        s.data.requires_grad_(True)
        s.xi.requires_grad_(True)
        return s
    if kind == "step":
        s.x, s.dx, s.d2x, s.c = g.x, g.dx, g.d2x, g.c
        return s
    s.plan = _plan(g, s.opt)
    if kind == "apply":
        s.op = OPS[c["op"]] | (L.LBF_OP_TRANSPOSE if c.get("transpose") else 0)
        if c["op"] == "density":
            s.vec = s.vec[:s.N].contiguous()
        s.out = torch.empty_like(s.vec)
    elif kind == "many":
        s.sigma, s.a = _empty(c["nrhs"], s.N), _empty(c["nrhs"], s.M)
        s.work = torch.empty(max(1, L.lbf_gmres_workspace_many(s.plan, c["nrhs"])),
                             dtype=torch.uint8, device=_dev())
    if kind in ("solve", "evaluate"):
        s.sigma, s.u = _empty(s.N), _empty(c["targets"])
        s.a = _empty(s.M) if s.M > 1 else None  # one island: its multiplier is zero
    if kind == "solve" and s.N <= 1 << 18:  # small solves: on a stream of their own
        s.stream = torch.cuda.Stream()
    else:
        s.stream = None
    return s


def _solve(s, plan, sigma, a, u):
    rc, _, _ = L.lbf_gmres_solve(plan, s.data, sigma, a)
    if rc != L.LBF_OK:
        raise L.LbfError(rc, "lbf_gmres_solve")
    L.lbf_evaluate(plan, sigma, a, s.targets, u)


def run(s):
    kind = s.case["kind"]
    if kind == "apply":
        L.lbf_apply(s.plan, s.op, s.vec, s.out)
        return s.out
    if kind == "evaluate":
        L.lbf_evaluate(s.plan, s.vec[:s.N], s.vec[s.N:], s.targets, s.u)
        return s.u
    if kind == "solve":
        if s.stream is None:
            _solve(s, s.plan, s.sigma, s.a, s.u)
        else:
            s.stream.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(s.stream):
                _solve(s, s.plan, s.sigma, s.a, s.u)
            torch.cuda.current_stream().wait_stream(s.stream)
        return {"sigma": s.sigma, "a": s.a, "u": s.u} if s.M > 1 else {"sigma": s.sigma, "u": s.u}
    if kind == "many":
        rc, _, _ = L.lbf_gmres_solve_many(s.plan, s.data, s.sigma, s.a, work=s.work)
        if rc != L.LBF_OK:
            raise L.LbfError(rc, "lbf_gmres_solve_many")
        return {"sigma": s.sigma, "a": s.a}
    if kind == "gradient":
        u = solve_evaluate(s.data, s.xi, s.dxi, s.d2xi, s.c, s.targets, s.ptr, s.opt)
        gd, gx = torch.autograd.grad((u * u).mean(), [s.data, s.xi])
        return {"u": u.detach(), "data": gd, "nodes": gx}
    if kind == "step":
        plan = L.lbf_plan_create(s.ptr, s.x, s.dx, s.d2x, s.c, opt=s.opt)
        sigma, a, u = _empty(s.N), _empty(s.M), _empty(s.case["targets"])
        _solve(s, plan, sigma, a, u)
        return {"sigma": sigma, "a": a, "u": u}
    res = L.lbf_batch_run(s.items, opt=s.opt, nworkers=8)
    if any(r["status"] != L.LBF_OK for r in res):
        raise RuntimeError("lbf_batch_run: " + str([r["status"] for r in res]))
    return [{k: r[k] for k in ("sigma", "a", "u")} for r in res]


# ---- the least work -----------------------------------------------------------------


def _apply_flops(N, P, leaf, direct):
    """A textbook FMM application: about two leaves of near pairs a node at 11 flops, P2M,
    L2P, 27 M2L a box over about 3 N / leaf boxes, and the shifts."""
    if direct:
        return 11.0 * N * N
    return N * (22.0 * leaf + 16.0 * P) + 3.0 * N / leaf * (27 * 4 + 4) * P * P


def work(case):
    c = case
    if c["kind"] == "batch":
        parts = [_work(dict(q, kind="many")) for q in _many_geometries(c)]
    else:
        parts = [_work(c)]
    return {k: float(sum(p[k] for p in parts)) for k in ("bytes", "flops")}


def _work(c):
    mean = c["lo"] if c["lo"] == c["hi"] else (c["hi"] - c["lo"]) / math.log(c["hi"] / c["lo"])
    N, M, P, T = c["M"] * mean, c["M"], c["p"] + 1, c.get("targets", 0)
    geo = 48.0 * N  # xi, w, self term, sphere correction
    one = _apply_flops(N, P, c["leaf"], c.get("direct"))
    kind = c["kind"]
    if kind == "apply":
        return {"bytes": geo + 16.0 * (N + M), "flops": one}
    if kind == "evaluate":
        return {"bytes": geo + 8.0 * (N + M) + 32.0 * T, "flops": T * (200.0 + 8 * P * 27)}
    if kind == "many":
        return {"bytes": geo + 16.0 * c["nrhs"] * (N + M), "flops": 15.0 * c["nrhs"] * one}
    if kind == "gradient":
        return {"bytes": 48.0 * N + 40.0 * N + 32.0 * T, "flops": 35.0 * one}
    setup = 72.0 * N if kind == "step" else geo
    return {"bytes": setup + 16.0 * (N + M) + 32.0 * T, "flops": 20.0 * one}


# ---- the same in plain 64-bit torch -------------------------------------------------
#
# From the 3D form of the equations: the double-layer kernel -(1/2 pi) (t - x).(x x x') /
# |t - x|^2 per unit parameter with its diagonal limit, G = -(1/4 pi) log(|t - c|^2 / 2),
# and the bordered matrix [[I + 2K, 2G], [F, D]] (F: the sums over islands 1..M-1, D: ones
# in the last row).


def _kernel_block(t, g, lo, hi):
    """h_j K(t_i, x_j), j in lo..hi."""
    x, n = g.x[lo:hi], torch.linalg.cross(g.x[lo:hi], g.dx[lo:hi]) * (g.h[lo:hi] / -TWO_PI)[:, None]
    num = den = None
    for k in range(3):
        d = t[:, k, None] - x[None, :, k]
        num = d * n[None, :, k] if num is None else num.addcmul_(d, n[None, :, k])
        den = d.mul_(d) if den is None else den.addcmul_(d, d)
    return num.div_(den)


def _diagonal(g):
    num = (g.x * torch.linalg.cross(g.dx, g.d2x)).sum(1)
    return -num / (2 * TWO_PI * (g.dx * g.dx).sum(1)) * g.h


def _double_layer(g, v, transpose):
    """2 K v (or its transpose) by blocks of rows."""
    out = torch.zeros_like(v)
    step = max(1, (1 << 27) // g.N)
    for a in range(0, g.N, step):
        b = min(g.N, a + step)
        k = _kernel_block(g.x[a:b], g, 0, g.N)
        k[torch.arange(b - a), torch.arange(a, b)] = 0.0
        if transpose:
            out += k.T @ v[a:b]
        else:
            out[a:b] = k @ v
    return 2 * (out + _diagonal(g) * v)


def _green(t, c):
    d = ((t[:, None, :] - c[None, :, :]) ** 2).sum(2)
    return (math.log(2.0) - torch.log(d)) / (2 * TWO_PI)


def _island_sums(g, v):
    """F v as an M-vector whose last entry (no constraint row) is 0."""
    s = torch.zeros(g.M, dtype=F64, device=v.device).index_add_(0, g.isl, v)
    return torch.cat([s[1:], s.new_zeros(1)])


def _island_spread(g, y):
    """F^T y."""
    return torch.cat([y.new_zeros(1), y[:-1]])[g.isl]


def _last_row(g, y):
    out = torch.zeros_like(y)
    out[-1] = y.sum()
    return out


def _exact_apply(c, g, vec):
    N, op, tr = g.N, c["op"], bool(c.get("transpose"))
    s, a = vec[:N], vec[N:]
    if op == "density":
        return s + _double_layer(g, s, tr)
    E = 2 * _green(g.x, g.c)
    S = -torch.stack([_island_sums(g, E[:, k]) for k in range(g.M)], 1)
    S[-1] += 1.0
    if op == "full" and not tr:
        return torch.cat([s + _double_layer(g, s, False) + E @ a, _island_sums(g, s) + _last_row(g, a)])
    if op == "full":
        return torch.cat([s + _double_layer(g, s, True) + _island_spread(g, a), E.T @ s + a[-1]])
    if not tr:  # P^-1 A [s; a] = [s + v + E y; a - y], v = 2 K s, S y = F v
        v = _double_layer(g, s, False)
        y = torch.linalg.solve(S, _island_sums(g, v))
        return torch.cat([s + v + E @ y, a - y])
    # P^-T A^T [s; a] = [s + w - F^T z; a + z], w = 2 K^T s, S^T z = -E^T w
    w = _double_layer(g, s, True)
    z = torch.linalg.solve(S.T, -(E.T @ w))
    return torch.cat([s + w - _island_spread(g, z), a + z])


def _exact_solve(g, data):
    """Dense solves for the columns of data (N x n): (sigma, a)."""
    A = torch.zeros(g.N + g.M, g.N + g.M, dtype=F64, device=data.device)
    K = _kernel_block(g.x, g, 0, g.N)
    K.fill_diagonal_(0.0)
    A[:g.N, :g.N] = 2 * K
    i = torch.arange(g.N, device=data.device)
    A[i, i] = 1 + 2 * _diagonal(g)
    A[:g.N, g.N:] = 2 * _green(g.x, g.c)
    on = g.isl > 0
    A[g.N + g.isl[on] - 1, i[on]] = 1.0
    A[-1, g.N:] = 1.0
    b = torch.cat([2 * data, data.new_zeros(g.M, data.shape[1])])
    z = torch.linalg.solve(A, b)
    return z[:g.N], z[g.N:]


def _exact_one(c, seed):
    g, m = _inputs(c, seed)
    kind = c["kind"]
    if kind == "apply":
        return _exact_apply(c, g, m["vec"]) if g.N <= 220_000 and g.M <= 2000 else None
    if kind == "evaluate":
        s, a, out = m["vec"][:g.N], m["vec"][g.N:], []
        step = max(1, (1 << 27) // g.N)
        for t in m["targets"].split(step):
            out.append(_kernel_block(t, g, 0, g.N) @ s + _green(t, g.c) @ a)
        return torch.cat(out)
    u = _pair_potential(m["targets"], m["src"]) if kind not in ("many", "batch") else None
    if kind == "gradient":
        return {"u": u if c["lo"] >= 256 else None, "data": None, "nodes": None}
    small = g.N + g.M <= 12000
    if kind in ("many", "batch"):
        if not small:
            return None
        sigma, a = (v.T.contiguous() for v in _exact_solve(g, m["data"].T))
        return {"sigma": sigma, "a": a, "u": None} if kind == "batch" else {"sigma": sigma, "a": a}
    if small:
        sigma, a = _exact_solve(g, m["data"][:, None])
        sigma, a = sigma[:, 0], a[:, 0]
        u = _kernel_block(m["targets"], g, 0, g.N) @ sigma + _green(m["targets"], g.c) @ a
        return {"sigma": sigma, "a": a if g.M > 1 else None, "u": u}
    # large: the pair's potential where the curves are resolved, no dense solution
    return {"sigma": None, "a": None, "u": u if c["lo"] >= 512 else None}


def exact(case, seed):
    if case["kind"] != "batch":
        return _exact_one(case, seed)
    got = [_exact_one(q, seed * 1000 + k) for k, q in enumerate(_many_geometries(case))]
    return [v if v is not None else {"sigma": None, "a": None, "u": None} for v in got]

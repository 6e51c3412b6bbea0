"""Performance cases of the fractional-Laplacian library: what users have it do, through its public entry points.

Kinds: "apply" (y = A u, single or batched), "sweep" (a plan for one alpha, its symbol and one apply), "solve"
(the fractional Poisson problem), "allen_cahn" (a batch of instances) and "learn" (one training step of the
learned preconditioner).  `exact` restates each in FP64 with plain torch: its own quadrature, coefficients and
circulant embedding, none of the library's code.
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

import paper_1804_02718_gb300 as fl

PREC = {"f64": fl.FRLAP_F64, "f32": fl.FRLAP_F32, "df64": fl.FRLAP_DF64, "mixed": fl.FRLAP_MIXED,
        "mixed_df64": fl.FRLAP_MIXED_DF64}
PRECOND = {"none": fl.FRLAP_PRECOND_NONE, "strang": fl.FRLAP_PRECOND_STRANG, "tau": fl.FRLAP_PRECOND_TAU}
SOLVER = {"cg": fl.FRLAP_SOLVE_CG, "ir": fl.FRLAP_SOLVE_IR}
AC_TAU, AC_EPS = 1e-3, 0.05  # the batched Allen-Cahn workload's step and interface width
F64 = torch.float64


def _apply(name, prec, alpha, N, batch=1, tuned=False):
    N = tuple(N) + (0,) * (3 - len(N))
    return dict(name=name, kind="apply", prec=prec, alpha=alpha, nx=N[0], ny=N[1], nz=N[2], batch=batch, tuned=tuned)


def _solve(name, prec, alpha, N, precond, solver):
    N = tuple(N) + (0,) * (3 - len(N))
    return dict(name=name, kind="solve", prec=prec, alpha=alpha, nx=N[0], ny=N[1], nz=N[2], precond=precond,
                solver=solver)


def listed():
    return [
        # a single call on a small rectangular grid in the default precision: launches and latency
        _apply("apply_2d_f64_small", "f64", 1.2, (100, 70)),
        # the headline workload: 8 vectors at 2047^2 in double-float, on a tuned plan
        _apply("apply_2d_df64_batch", "df64", 1.5, (2048, 2048), 8, True),
        # the same throughput workload in FP32 (inner solves and preconditioners run this engine)
        _apply("apply_2d_f32_batch", "f32", 1.5, (2048, 2048), 8, True),
        # one vector on a ragged grid, untuned: what a Krylov loop of the caller's own does
        _apply("apply_2d_df64_ragged", "df64", 0.8, (1500, 1100)),
        # an alpha sweep at a table's mesh size: plan, symbol and one apply in native FP64
        dict(name="sweep_2d_f64", kind="sweep", prec="f64", alpha=0.7, nx=512, ny=512, nz=0),
        # the 3D throughput workload
        _apply("apply_3d_df64_batch", "df64", 1.0, (256, 256, 256), 2, True),
        # one FP32 vector on a ragged box, untuned
        _apply("apply_3d_f32_ragged", "f32", 1.0, (250, 220, 190)),
        # the solver headline: 2047^2 to 1e-10 with the sine-basis preconditioner
        _solve("solve_2d_tau", "df64", 1.5, (2048, 2048), "tau", "cg"),
        # a small plain CG solve in the default precision: latency of the solver loop
        _solve("solve_2d_cg_small", "f64", 1.5, (128, 128), "none", "cg"),
        # FP32-inner iterative refinement in 3D
        _solve("refine_3d_tau", "mixed_df64", 1.0, (128, 128, 128), "tau", "ir"),
        # batched semi-implicit Allen-Cahn: instances on 255^2, 511^2 and 1023^2 grids
        dict(name="allen_cahn_batch", kind="allen_cahn", prec="df64", count=12, n0=256, n1=512, n2=1024, steps=4),
        # one training step (gradient and Adam) of the learned preconditioner at its training grid
        dict(name="learn_step", kind="learn", prec="f64", alpha=1.3, nx=256, ny=256, nz=0, batch=8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "sweep", "solve", "solve", "allen_cahn", "learn"])
    alpha = round(rng.uniform(0.5, 1.9), 3)
    if kind == "apply":
        prec = rng.choice(["f64", "f32", "df64"])
        if rng.random() < 0.6:
            hi = 1024 if prec == "f64" else 2048
            N = (_log_int(rng, 12, hi), _log_int(rng, 12, hi))
            batch = rng.choice([1, 1, 2, 3, 8])
        else:
            hi = 128 if prec == "f64" else 256
            N = tuple(_log_int(rng, 8, hi) for _ in range(3))
            batch = rng.choice([1, 1, 2])
        return {k: v for k, v in _apply("", prec, alpha, N, batch, rng.random() < 0.3).items() if k != "name"}
    if kind == "sweep":
        return dict(kind=kind, prec=rng.choice(["f64", "df64"]), alpha=alpha, nx=_log_int(rng, 16, 600),
                    ny=_log_int(rng, 16, 600), nz=0)
    if kind == "solve":
        solver = rng.choice(["cg", "ir"])
        prec = rng.choice(["mixed", "mixed_df64"]) if solver == "ir" else rng.choice(["f64", "df64"])
        d = rng.choice([2, 2, 3])
        precond = rng.choice(["none", "strang", "tau"])
        if precond == "tau":  # powers of two
            N = tuple(2 ** rng.randint(5, 10 if d == 2 else 7) for _ in range(d))
        else:
            N = tuple(_log_int(rng, 24, 256 if d == 2 else 64) for _ in range(d))
        if precond == "none":
            alpha = min(alpha, 1.5)
        return {k: v for k, v in _solve("", prec, alpha, N, precond, solver).items() if k != "name"}
    if kind == "allen_cahn":
        return dict(kind=kind, prec=rng.choice(["f64", "df64"]), count=rng.randint(1, 9), n0=_log_int(rng, 32, 256),
                    n1=_log_int(rng, 64, 512), n2=_log_int(rng, 64, 512), steps=rng.randint(1, 4))
    d3 = rng.random() < 0.3
    hi = 48 if d3 else 256
    return dict(kind=kind, prec="f64", alpha=alpha, nx=_log_int(rng, 20, hi), ny=_log_int(rng, 20, hi),
                nz=_log_int(rng, 20, hi) if d3 else 0, batch=rng.randint(1, 8))


# ------------------------------------------------------------------------------------------- inputs
def _grid(case):
    return tuple(case[k] for k in ("nx", "ny", "nz") if case[k])


def _shape(N):
    return tuple(v - 1 for v in reversed(N))


def _h(N):
    return 2.0 / max(N)


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _gaussian_sum(N, seed, count=16):
    """sum_g A_g exp(-|x - c_g|^2 / (2 w_g^2)) on the interior nodes of the box with lower corner (-1, ..)."""
    rng = np.random.default_rng(seed)
    d, h = len(N), _h(N)
    centres, widths, amps = rng.uniform(-1.0, 1.0, (count, d)), rng.uniform(0.1, 0.4, count), rng.standard_normal(count)
    axes = [-1.0 + h * torch.arange(1, n, dtype=F64, device="cuda") for n in N]
    f = torch.zeros(_shape(N), dtype=F64, device="cuda")
    for g in range(count):
        e = torch.full((1,) * d, amps[g], dtype=F64, device="cuda")
        for r in range(d):  # axis r is dimension d - 1 - r (x fastest)
            shape = [1] * d
            shape[d - 1 - r] = -1
            e = e * torch.exp(-(axes[r] - centres[g, r]) ** 2 / (2.0 * widths[g] ** 2)).reshape(shape)
        f += e
    return f


def _ac_instances(case, seed):
    """(N, alpha, u0) of every instance: alpha ~ U[1.2, 1.9], u0 ~ U[-0.9, 0.9], grids in turn."""
    alphas = np.random.default_rng(seed).uniform(1.2, 1.9, size=case["count"])
    g = _gen(seed)
    out = []
    for i in range(case["count"]):
        n = case["n%d" % (i % 3)]
        u = 1.8 * torch.rand((n - 1, n - 1), dtype=F64, device="cuda", generator=g) - 0.9
        out.append((n, float(alphas[i]), u))
    return out


def _learn_inputs(case, seed):
    """Errors e (smooth fields with a rough part, as CG's are) and network parameters in training."""
    N = _grid(case)
    g = _gen(seed)
    e = torch.stack([_gaussian_sum(N, seed + 17 * b) for b in range(case["batch"])])
    e += 0.02 * torch.randn(e.shape, dtype=F64, device="cuda", generator=g)
    rng = np.random.default_rng(seed)
    H = 64
    parts = [0.3 * rng.standard_normal(4 * H), 0.1 * rng.standard_normal(H),
             0.3 / math.sqrt(H) * rng.standard_normal(H * H), 0.1 * rng.standard_normal(H),
             0.05 * rng.standard_normal(H), 0.05 * rng.standard_normal(1)]
    params = torch.from_numpy(np.concatenate(parts).astype(np.float32)).cuda()
    m1 = torch.from_numpy((1e-3 * rng.standard_normal(params.numel())).astype(np.float32)).cuda()
    m2 = torch.from_numpy((1e-6 * (0.5 + rng.random(params.numel()))).astype(np.float32)).cuda()
    return e, params, m1, m2


def _apply_input(case, seed):
    N = _grid(case)
    dt = torch.float32 if case["prec"] == "f32" else F64
    shape = (case.get("batch", 1),) + _shape(N)
    return torch.randn(shape, dtype=dt, device="cuda", generator=_gen(seed))


def _bytes(nbytes):
    raw = torch.empty(nbytes + 256, dtype=torch.uint8, device="cuda")
    off = (-raw.data_ptr()) % 256
    return raw[off:off + nbytes]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "allen_cahn":
        inst = _ac_instances(case, seed)
        plans = [fl.Plan(2, a, 2.0 / n, (n, n), prec=PREC[case["prec"]]) for n, a, _ in inst]
        work = _bytes(fl.frlap_allen_cahn_batch_workspace_bytes(plans))
        return dict(kind=kind, plans=plans, u0=[u for _, _, u in inst], steps=case["steps"], work=work)
    N = _grid(case)
    d, h = len(N), _h(N)
    if kind == "sweep":
        return dict(kind=kind, args=(d, case["alpha"], h, N), prec=PREC[case["prec"]],
                    u=_apply_input(case, seed).reshape(_shape(N)))
    plan = fl.Plan(d, case["alpha"], h, N, prec=PREC[case["prec"]])
    if kind == "apply":
        u = _apply_input(case, seed)
        batch = case["batch"]
        if case["tuned"]:
            fl.frlap_plan_autotune(plan, batch)
        work = _bytes(fl.frlap_apply_batch_workspace_bytes(plan, batch))
        return dict(kind=kind, plan=plan, u=u, y=torch.empty_like(u), batch=batch, work=work)
    if kind == "solve":
        if case["precond"] == "tau":
            fl.frlap_precond_tau(plan)
        elif case["precond"] == "strang":
            fl.frlap_precond_strang(plan)
        return dict(kind=kind, plan=plan, f=_gaussian_sum(N, seed), precond=PRECOND[case["precond"]],
                    solver=SOLVER[case["solver"]])
    e, params, m1, m2 = _learn_inputs(case, seed)
    r = torch.empty_like(e)
    fl.frlap_apply_batch(plan, e, r)
    return dict(kind=kind, plan=plan, e=e, r=r, params=params, m1=m1, m2=m2,
                work=_bytes(fl.frlap_learn_workspace_bytes(plan, case["batch"])))


def run(s):
    kind = s["kind"]
    if kind == "apply":
        if s["batch"] > 1:
            return fl.frlap_apply_batch(s["plan"], s["u"], s["y"], work=s["work"])
        return fl.frlap_apply(s["plan"], s["u"], s["y"], work=s["work"])
    if kind == "sweep":
        plan = fl.Plan(*s["args"], prec=s["prec"])
        out = fl.frlap_apply(plan, s["u"]), plan.symbol()
        plan.close()
        return out
    if kind == "solve":
        return fl.frlap_pcg_solve(s["plan"], s["f"], solver=s["solver"], precond=s["precond"])[0]
    if kind == "allen_cahn":
        us = [u.clone() for u in s["u0"]]
        fl.frlap_allen_cahn_batch(s["plans"], us, AC_TAU, AC_EPS, s["steps"], work=s["work"])
        return us
    params, m1, m2 = s["params"].clone(), s["m1"].clone(), s["m2"].clone()
    grad, loss = torch.empty_like(params), torch.empty(1, dtype=F64, device="cuda")
    fl.frlap_learn_grad(s["plan"], params, s["r"], s["e"], grad, loss, s["work"])
    fl.frlap_adam_step(params, grad, m1, m2, 2e-3, 10)
    return grad, loss, params, m1, m2


# ------------------------------------------------------------------------------------------- work
def _pow2(n):
    return max(32, 1 << (2 * (n - 1) - 2).bit_length())


def _apply_work(N, real_bytes, batch=1):
    """One input and one output vector each, and the symbol octant once; the padded transforms' flops (the
    zero and the cropped halves of the lines left out)."""
    n = [v - 1 for v in N]
    P = [_pow2(v) for v in N]
    M = math.prod(n)
    nbytes = 2 * M * real_bytes * batch + math.prod(p // 2 + 1 for p in P) * real_bytes
    flops = 2 * math.prod(n[1:]) * 2.5 * P[0] * (math.log2(P[0]) - 1)
    flops += 2 * (P[0] // 2 + 1) * (n[2] if len(N) == 3 else 1) * 5 * P[1] * (math.log2(P[1]) - 1)
    if len(N) == 3:
        flops += 2 * (P[0] // 2 + 1) * P[1] * 5 * P[2] * (math.log2(P[2]) - 1)
    return nbytes, flops * batch


def work(case):
    kind = case["kind"]
    eb = 4 if case["prec"] == "f32" else 8
    if kind == "allen_cahn":
        b = f = 0.0
        for i in range(case["count"]):
            n = case["n%d" % (i % 3)]
            wb, wf = _apply_work((n, n), eb)
            its = 6 * case["steps"]  # CG iterations of a step at this step size, about
            b, f = b + its * wb, f + its * wf
        return {"bytes": b, "flops": f}
    N = _grid(case)
    wb, wf = _apply_work(N, eb, case.get("batch", 1))
    if kind == "apply":
        return {"bytes": wb, "flops": wf}
    if kind == "sweep":  # the coefficients' quadrature: 16 to 400 powers per element, a dozen flops each
        return {"bytes": wb, "flops": wf + 8 * 25 * math.prod(N)}
    if kind == "solve":
        its = {"tau": 12, "strang": 40}.get(case["precond"], int(2 * max(N) ** (case["alpha"] / 2)))
        return {"bytes": its * 1.5 * wb, "flops": its * 1.5 * wf}
    entries = math.prod(_pow2(v) // 2 + 1 for v in N)
    return {"bytes": 2 * wb, "flops": 3 * wf + 6 * 4545 * entries}


# ------------------------------------------------------------------------------------------- exact values
def _rule(q):
    x, w = np.polynomial.legendre.leggauss(q)
    return (torch.tensor(0.5 * (x + 1.0), dtype=F64, device="cuda"), torch.tensor(0.5 * w, dtype=F64, device="cuda"))


def _elements(lo, K, d, p, q):
    """int over [k, k+1] of |xi|^-p for lower corners k with k_0 in lo, the others in [0, K)."""
    x, w = _rule(q)
    t = torch.arange(K, dtype=F64, device="cuda")
    a = (lo.to(F64)[:, None] + x) ** 2
    b = (t[:, None] + x) ** 2
    if d == 2:
        r2 = a[:, :, None, None] + b
        return torch.einsum("aibj,i,j->ab", r2 ** (-p / 2), w, w)
    r2 = a[:, :, None, None, None, None] + b[:, :, None, None] + b
    return torch.einsum("aibjcl,i,j,l->abc", r2 ** (-p / 2), w, w, w)


def _coefficients(d, alpha, h, N):
    """a_k for k in [0, N]^d (gamma = 2) from tensor Gauss-Legendre element integrals, with the origin element
    and the far field by a pyramid split."""
    p = d + alpha - 2.0
    w = torch.empty((N,) * d, dtype=F64, device="cuda")
    step = N if d == 2 and N <= 256 else max(1, 2 ** (26 if d == 2 else 24) // (N ** (d - 1) * 5 ** d // 4))
    for s in range(0, N, step):
        w[s:s + step] = _elements(torch.arange(s, min(s + step, N), device="cuda"), N, d, p, 5)
    for K, q in ((48, 8), (12, 14), (3, 24)):  # nearer elements: more points
        K = min(K + 1, N)
        for s in range(K):
            w[(slice(s, s + 1),) + (slice(0, K),) * (d - 1)] = _elements(torch.tensor([s], device="cuda"), K, d, p, q)
    x, wq = _rule(40)
    s2, ws = (x * x, wq) if d == 2 else ((x * x)[:, None] + x * x, wq[:, None] * wq)
    w0 = d / (d - p) * (ws * (1.0 + s2) ** (-p / 2)).sum()
    far = d * float(N) ** (-alpha) / alpha * (ws * (1.0 + s2) ** (-(d + alpha) / 2)).sum()
    w[(0,) * d] = w0
    a = torch.zeros((N + 1,) * d, dtype=F64, device="cuda")
    for e in itertools.product((0, 1), repeat=d):  # the elements that have k as a vertex
        a[tuple(slice(v, N + v) for v in e)] += w
    del w
    for v in itertools.product((0, 1), repeat=d):  # origin correction on the unit vertices
        if sum(v):
            a[v] += ((2.0 if d == 2 else 8.0 / 3.0) if sum(v) == 1 else 0.0) * w0 - w0
    t = torch.arange(N + 1, dtype=F64, device="cuda")
    for r in range(d):  # 2^sigma / 2^d: halves along each non-zero coordinate
        a[(slice(None),) * r + (slice(1, None),)] *= 0.5
    k2 = sum((t * t).reshape([-1 if i == r else 1 for i in range(d)]) for r in range(d))
    a[(0,) * d] = 0.0
    a /= torch.where(k2 > 0, k2, torch.ones_like(k2))
    del k2
    m = torch.where(t > 0, 2.0, 1.0).to(F64)
    tot = a
    for _ in range(d):
        tot = tot @ m
    a[(0,) * d] = -tot - 2.0 ** d * far
    return a * h ** (-alpha)


class _Operator:
    """A of one case in FP64: circulant embedding of P points per axis with torch's FFT."""

    def __init__(self, N, alpha, h=None):
        d = len(N)
        h = _h(N) if h is None else h
        n = [v - 1 for v in N]
        c = (2.0 ** (alpha - 1.0) * alpha * math.gamma((d + alpha) / 2.0)
             / (math.pi ** (d / 2.0) * math.gamma(1.0 - alpha / 2.0)))
        coef = _coefficients(d, alpha, h, max(N))
        self.shape, self.P = _shape(N), tuple(_pow2(v) for v in reversed(N))
        g = torch.zeros(self.P, dtype=F64, device="cuda")
        idx = []
        for r in range(d):
            k = torch.arange(self.P[r], device="cuda")
            f = torch.minimum(k, self.P[r] - k)
            idx.append((k[f < self.shape[r]], f[f < self.shape[r]]))
        pos = torch.meshgrid(*[i for i, _ in idx], indexing="ij")
        mag = torch.meshgrid(*[j for _, j in idx], indexing="ij")
        g[pos] = -c * coef[mag]
        del pos, mag, coef
        self.lam = torch.fft.rfftn(g).real
        self.d = d
        self.dims = tuple(range(-d, 0))

    def mult(self, u, m):
        U = torch.fft.rfftn(u, s=self.P, dim=self.dims)
        y = torch.fft.irfftn(U * m, s=self.P, dim=self.dims)
        return y[tuple(slice(0, v) for v in self.shape)].contiguous()

    def __call__(self, u):
        return self.mult(u, self.lam)

    def octant(self):
        return self.lam[tuple(slice(0, p // 2 + 1) for p in self.P)].contiguous()


def _pcg(apply, f, x, precond=None, rtol=1e-14, maxit=400):
    """Preconditioned CG in FP64, on from x until the recursive residual is rtol ||f||."""
    r = f - apply(x) if x is not None else f.clone()
    x = torch.zeros_like(f) if x is None else x.clone()
    z = precond(r) if precond else r
    p = z.clone()
    rz = (r * z).sum()
    stop = float((f * f).sum()) * rtol * rtol
    for _ in range(maxit):
        if float((r * r).sum()) <= stop:
            break
        q = apply(p)
        al = rz / (p * q).sum()
        x += al * p
        r -= al * q
        z = precond(r) if precond else r
        new = (r * z).sum()
        p = z + (new / rz) * p
        rz = new
    return x


def _exact_learn(case, seed):
    N = _grid(case)
    e, params, m1, m2 = _learn_inputs(case, seed)
    op = _Operator(N, case["alpha"])
    th = params.double().requires_grad_(True)
    H = 64
    W1, b1, W2, b2, w3, b3 = torch.split(th, [4 * H, H, H * H, H, H, 1])
    axes = [torch.arange(p // 2 + 1, dtype=F64, device="cuda") / (p // 2) for p in op.P]
    kap = list(reversed([t.reshape(-1) for t in torch.meshgrid(*axes, indexing="ij")]))
    phi = torch.zeros(kap[0].numel(), 4, dtype=F64, device="cuda")
    phi[:, 0] = float(np.float32(case["alpha"]))
    for r, k in enumerate(kap):
        phi[:, 1 + r] = k
    h1 = torch.tanh(phi @ W1.reshape(H, 4).T + b1)
    h2 = torch.tanh(h1 @ W2.reshape(H, H).T + b2)
    lam = op.octant()
    m = torch.exp(h2 @ w3 + b3).reshape(lam.shape) / lam
    half = m  # unfold the octant to rfftn's half spectrum: even along every axis but the last
    for ax, p in enumerate(op.P[:-1]):
        k = torch.arange(p, device="cuda")
        half = half.index_select(ax, torch.minimum(k, p - k))
    loss = 0.0
    for b in range(case["batch"]):
        r = op(e[b])
        z = op.mult(r, half)
        loss = loss + (1.0 + (-2.0 * (r * z).sum() + (z * op(z)).sum()) / (r * e[b]).sum()) / case["batch"]
    g, = torch.autograd.grad(loss, th)
    lr, be1, be2, eps = (float(np.float32(v)) for v in (2e-3, 0.9, 0.999, 1e-8))  # FP32 arguments
    t = 10
    n1 = be1 * m1.double() + (1 - be1) * g
    n2 = be2 * m2.double() + (1 - be2) * g * g
    new = params.double() - lr * (n1 / (1 - be1 ** t)) / (torch.sqrt(n2 / (1 - be2 ** t)) + eps)
    return g, loss.detach().reshape(1), new, n1, n2


def exact(case, seed):
    kind = case["kind"]
    if kind == "allen_cahn":
        out = []
        s = AC_TAU * AC_EPS ** 2
        for n, alpha, u in _ac_instances(case, seed):
            op = _Operator((n, n), alpha)
            for _ in range(case["steps"]):
                u = _pcg(lambda v: v + s * op(v), u + AC_TAU * (u - u ** 3), u)
            out.append(u)
        return out
    if kind == "learn":
        return _exact_learn(case, seed)
    N = _grid(case)
    op = _Operator(N, case["alpha"])
    if kind == "solve":
        return _pcg(op, _gaussian_sum(N, seed), None, lambda r: op.mult(r, 1.0 / op.lam))
    u = _apply_input(case, seed).double()
    if kind == "apply":
        return torch.stack([op(v) for v in u])
    scale = 1.0 / math.prod(op.P)  # the library's symbol carries the inverse transform's factor
    return op(u.reshape(_shape(N))), op.octant() * scale

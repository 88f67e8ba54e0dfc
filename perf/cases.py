"""Timed cases of the framework's public entry points.

Each case is one pass of a user's program: assembling an operator and applying
it, factoring and solving in the three storage forms, solving again with a
factorisation that is kept, differentiating a solve, and refactoring a batch of
operators.  Grids, truncation thresholds, admissibility, leaf sizes and rank
caps are those of the workload recipes, the tests and the benchmark, scaled
over the sizes whose planes the block structure supports (leaves of 25 to 64
points).  Every solve runs to a relative residual of 1e-10 or below, so that its
solution is determined by the operator and not by where the iteration stopped.
"""
import math

import torch

import paper_1712_08872_gb300 as acr

_PREC = {"fp64": acr.ACR_FP64, "fp32": acr.ACR_FP32, "bf16": acr.ACR_BF16}
_BYTES = {"fp64": 8, "fp32": 4, "bf16": 2}
_DEV = "cuda"


def listed():
    return [
        # the smallest call: assemble a small diffusion operator and multiply with it once
        # (an assembly step of a time loop, a residual check); launch latency
        {"name": "operator_n20", "kind": "operator", "pde": "poisson", "n": 20, "nrhs": 1},
        # the same on a full-size, odd grid and a few vectors: streaming through memory
        {"name": "operator_n127_rhs4", "kind": "operator", "pde": "codi", "n": 127, "nrhs": 4},
        # the small accurate solve of the Gaussian-field recipe (eps 1e-6, eta 1, leaf 32)
        {"name": "solve_grf_n16_fp64", "kind": "solve", "pde": "poisson", "n": 16, "prec": "fp64",
         "eps": 1e-6, "eta": 1.0, "leaf": 32, "cap": 32, "rtol": 1e-10},
        # the plain FP64 form, which the mixed form is compared with
        {"name": "solve_codi_n32_fp64", "kind": "solve", "pde": "codi", "n": 32, "prec": "fp64",
         "eps": 1e-2, "eta": 2.0, "leaf": 64, "cap": 24, "rtol": 1e-10},
        # the benchmark's own step (assemble, factor, GMRES) at half its grid width
        {"name": "solve_codi_n64_fp32", "kind": "solve", "pde": "codi", "n": 64, "prec": "fp32",
         "eps": 1e-2, "eta": 2.0, "leaf": 64, "cap": 24, "rtol": 1e-10},
        # the largest factorisation: a grid whose leaves are ragged (50 points, not 64)
        {"name": "solve_codi_n80_fp32", "kind": "solve", "pde": "codi", "n": 80, "prec": "fp32",
         "eps": 1e-2, "eta": 2.0, "leaf": 64, "cap": 24, "rtol": 1e-10},
        # BF16-stored factors on a diffusion problem with 49-point leaves
        {"name": "solve_grf_n56_bf16", "kind": "solve", "pde": "poisson", "n": 56, "prec": "bf16",
         "eps": 1e-2, "eta": 2.0, "leaf": 64, "cap": 24, "rtol": 1e-10},
        # a differentiable solve: forward, adjoint, gradients of the coefficient field and of f
        {"name": "gradient_grf_n48", "kind": "gradient", "n": 48, "rtol": 1e-10},
        # the indefinite operator's many right-hand sides with one kept factorisation
        {"name": "resolve_helmholtz_n64_rhs32", "kind": "resolve", "pde": "helmholtz", "n": 64,
         "prec": "fp32", "eps": 1e-5, "eta": 2.0, "leaf": 64, "cap": 48, "rtol": 1e-12,
         "nrhs": 32},
        # one more right-hand side with a kept factorisation (a time step, a Newton step)
        {"name": "resolve_codi_n96_fp32", "kind": "resolve", "pde": "codi", "n": 96,
         "prec": "fp32", "eps": 1e-2, "eta": 2.0, "leaf": 64, "cap": 24, "rtol": 1e-10,
         "nrhs": 1},
        # a few right-hand sides with the half-size factors
        {"name": "resolve_grf_n64_bf16_rhs8", "kind": "resolve", "pde": "poisson", "n": 64,
         "prec": "bf16", "eps": 1e-2, "eta": 2.0, "leaf": 64, "cap": 24, "rtol": 1e-10,
         "nrhs": 8},
        # a batch of small problems whose coefficients change: assemble, refactor, solve each
        {"name": "batch_grf_n32_n40_x3", "kind": "batch", "sizes": "32,40,32,40,32,40",
         "eps": 1e-2, "eta": 2.0, "leaf": 64, "cap": 24, "rtol": 1e-10},
    ]


def draw(rng):
    kind = rng.choice(["operator", "solve", "solve", "solve", "gradient", "resolve", "resolve",
                       "batch"])
    if kind == "operator":
        return {"kind": kind, "pde": rng.choice(["poisson", "codi", "helmholtz"]),
                "n": round(math.exp(rng.uniform(math.log(12), math.log(127)))),
                "nrhs": rng.randint(1, 4)}
    tol = {"eps": 1e-2, "eta": 2.0, "leaf": 64, "cap": rng.choice([20, 24, 28, 32]),
           "rtol": 1e-10}
    if kind == "batch":
        sizes = sorted(rng.choice([12, 16, 20, 24, 28, 32, 40]) for _ in range(rng.randint(2, 6)))
        return {"kind": kind, "sizes": ",".join(map(str, sizes)), **tol}
    if kind == "gradient":
        return {"kind": kind, "n": rng.choice([12, 16, 20, 24, 28, 32, 40, 48]),
                "rtol": rng.choice([1e-10, 3e-11, 1e-11])}
    prec = rng.choice(["fp32", "fp32", "bf16", "fp64"])
    if kind == "solve":
        n = rng.choice([12, 16, 20, 24, 28, 32] if prec == "fp64" else
                       [12, 16, 20, 24, 28, 32, 40, 48, 56, 64, 80])
        return {"kind": kind, "pde": rng.choice(["poisson", "codi"]), "n": n, "prec": prec, **tol}
    n = rng.choice([16, 24, 28, 32] if prec == "fp64" else [16, 24, 32, 40, 48, 56, 64, 80])
    # (the indefinite operator keeps the small eps and the rank cap of its recipe)
    pde = rng.choice(["poisson", "codi", "helmholtz"] if prec != "bf16" else ["poisson", "codi"])
    if pde == "helmholtz":
        n = min(n, 64)
        tol.update(eps=1e-5, rtol=1e-12, cap=48)
    return {"kind": kind, "pde": pde, "n": n, "prec": prec, **tol,
            "nrhs": rng.choice([1, 1, 2, 3, 5, 8, 16, 32])}


# ------------------------------------------------------------------ inputs
def _nodes(n):
    t = (torch.arange(n, dtype=torch.float64, device=_DEV) + 1.0) / (n + 1)
    return t


def _grf_kappa(n, gen):
    """exp of a Gaussian random field with squared-exponential covariance of
    length 0.2 and unit variance (the covariance factorises over the axes)."""
    t = _nodes(n).cpu()
    k = torch.exp(-((t[:, None] - t[None, :]) ** 2) / (2.0 * 0.2 ** 2))
    w, q = torch.linalg.eigh(k)
    s = ((q * w.clamp_min(0.0).sqrt()) @ q.T).to(_DEV)
    xi = torch.randn(n, n, n, dtype=torch.float64, device=_DEV, generator=gen)
    g = torch.einsum("ai,ijk->ajk", s, xi)
    g = torch.einsum("bj,ajk->abk", s, g)
    return torch.exp(torch.einsum("ck,abk->abc", s, g)).reshape(-1).contiguous()


def _uniform(gen, lo, hi, count):
    r = torch.rand(count, dtype=torch.float64, device=_DEV, generator=gen)
    return lo + (hi - lo) * r


def _codi_beta(n, gen):
    """beta = b (1,1,1)(1 + 0.5 sin 2 pi (x + a) sin 2 pi (y + c)), b near 50."""
    b, a, c = _uniform(gen, 0.0, 1.0, 3).tolist()
    t = _nodes(n)
    s = torch.sin(2 * math.pi * (t[None, :] + a)) * torch.sin(2 * math.pi * (t[:, None] + c))
    s = (45.0 + 10.0 * b) * (1.0 + 0.5 * s)                    # (y, x)
    return s[None, None].expand(3, n, n, n).reshape(-1).contiguous()


def _layers_sigma(n, gen):
    """(omega / c)^2 of a medium of 8 slabs normal to x, c in [1, 3], 10 grid
    spacings per wavelength at c = 1."""
    cuts = _uniform(gen, 0.0, 1.0, 7).sort().values
    c = _uniform(gen, 1.0, 3.0, 8)[torch.searchsorted(cuts, _nodes(n))]
    sig = (2.0 * math.pi * (n + 1) / 10.0 / c) ** 2
    return sig.expand(n, n, n).reshape(-1).contiguous()


_FIELD = {"poisson": _grf_kappa, "codi": _codi_beta, "helmholtz": _layers_sigma}
_STENCIL = {"poisson": acr.acr_stencil_poisson, "codi": acr.acr_stencil_codi,
            "helmholtz": acr.acr_stencil_helmholtz}


def _gen(seed):
    g = torch.Generator(device=_DEV)
    g.manual_seed(seed)
    return g


def _fields(case, seed):
    """The coefficient fields and right-hand sides of a case."""
    gen = _gen(seed)
    if case["kind"] == "batch":
        ns = [int(s) for s in case["sizes"].split(",")]
        return [(_grf_kappa(n, gen), _uniform(gen, -1.0, 1.0, n ** 3)) for n in ns]
    n = case["n"]
    field = _FIELD[case.get("pde", "poisson")](n, gen)
    return field, _uniform(gen, -1.0, 1.0, case.get("nrhs", 1) * n ** 3)


def _method(pde):
    return acr.ACR_PCG if pde == "poisson" else acr.ACR_GMRES


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        fields = _fields(case, seed)
        ns = [int(s) for s in case["sizes"].split(",")]
        coefs = []
        for n, (kappa, _) in zip(ns, fields):
            coefs.append(torch.empty(7 * n ** 3, dtype=torch.float64, device=_DEV))
            acr.acr_stencil_poisson(n, kappa, coefs[-1])
        batch = _Batch(ns, coefs, case)
        return {"case": case, "ns": ns, "fields": fields, "coefs": coefs, "batch": batch}
    field, f = _fields(case, seed)
    n = case["n"]
    state = {"case": case, "field": field, "f": f}
    if kind == "gradient":
        # dL/du of a loss 0.5 ||u - u_obs||^2 against a smooth observation, near the
        # solution's own size, so that forward and adjoint carry the same weight
        state["g"] = _uniform(_gen(seed + 1000003), -1.0, 1.0, n ** 3)
    if kind == "resolve":
        coef = torch.empty(7 * n ** 3, dtype=torch.float64, device=_DEV)
        _STENCIL[case["pde"]](n, field, coef)
        state["coef"] = coef
        state["handle"] = acr.Handle(n, coef, case["eps"], case["eta"], case["leaf"],
                                     _PREC[case["prec"]], case["cap"])
    return state


class _Batch:
    """Owner of a batch pointer."""

    def __init__(self, ns, coefs, case):
        self.ptr = acr.acr_batch_create(ns, coefs, case["eps"], case["eta"], case["leaf"],
                                        acr.ACR_FP32, case["cap"])

    def __del__(self):
        try:
            acr.acr_batch_destroy(self.ptr)
        except Exception:
            pass


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "batch":
        for n, (kappa, _), coef in zip(state["ns"], state["fields"], state["coefs"]):
            acr.acr_stencil_poisson(n, kappa, coef)
        b = state["batch"].ptr
        acr.acr_batch_refactor(b)
        acr.acr_batch_status(b)
        out = []
        for i, (n, (_, f), coef) in enumerate(zip(state["ns"], state["fields"], state["coefs"])):
            u = torch.zeros(n ** 3, dtype=torch.float64, device=_DEV)
            acr.acr_batch_krylov_solve(b, i, coef, acr.ACR_PCG, 30, case["rtol"], 200, f, u)
            out.append(u)
        return out
    n, f = case["n"], state["f"]
    if kind == "gradient":
        kappa = state["field"].clone().requires_grad_(True)
        rhs = f.clone().requires_grad_(True)
        u = acr.acr_poisson_solve(kappa, rhs, rtol=case["rtol"])
        u.backward(state["g"])
        return {"u": u.detach(), "kappa": kappa.grad, "f": rhs.grad}
    if kind == "resolve":
        u = torch.zeros_like(f)
        acr.acr_krylov_solve(state["handle"].h, state["coef"], _method(case["pde"]), 30,
                             case["rtol"], 200, f, u, nrhs=case["nrhs"])
        return u
    coef = torch.empty(7 * n ** 3, dtype=torch.float64, device=_DEV)
    _STENCIL[case["pde"]](n, state["field"], coef)
    if kind == "operator":
        y = torch.empty_like(f)
        acr.acr_spmv(n, coef, f, y, case["nrhs"])
        return {"coef": coef, "y": y}
    h = acr.Handle(n, coef, case["eps"], case["eta"], case["leaf"], _PREC[case["prec"]],
                   case["cap"])
    u = torch.zeros_like(f)
    acr.acr_krylov_solve(h.h, coef, _method(case["pde"]), 30, case["rtol"], 200, f, u)
    h.close()
    return u


# ------------------------------------------------------------------ work
_counts = {}


def _leaf_counts(n, eta, leaf):
    """(dense leaves, points per leaf, low-rank rows + columns) of a plane block."""
    key = (n, eta, leaf)
    if key not in _counts:
        c, _, _ = acr.acr_structure_query(n, eta, leaf)
        size = n * n
        while size > leaf:
            size //= 2
        _counts[key] = (c[1], size, c[3] + c[4])
    return _counts[key]


# mean rank of the stored low-rank blocks, by the truncation threshold
def _rank(eps):
    return 3.0 if eps > 1e-4 else 6.0


def _factor_entries(n, eta, leaf, eps):
    nd, lsz, rows = _leaf_counts(n, eta, leaf)
    return nd * lsz * lsz + rows * _rank(eps)


def _setup_work(n, eta, leaf, eps, width):
    """A lower estimate of one factorisation: the stored factors (about 3 n plane
    H-matrices) written once, and per plane block the dense leaf products that an
    H-inverse and the Schur updates cannot do without."""
    nd, lsz, _ = _leaf_counts(n, eta, leaf)
    chunks = max(1, (n * n) // lsz)
    per_row = nd / chunks                                   # dense leaves of a block row
    product = 2.0 * chunks * per_row * per_row * lsz ** 3   # one H x H product's dense part
    return {"bytes": 56.0 * n ** 3 + 3.0 * n * _factor_entries(n, eta, leaf, eps) * width,
            "flops": n * 6.0 * product}


def _solve_work(n, eta, leaf, eps, width, nrhs, iterations):
    """Each iteration reads the stored factors once (the inverses twice) and the
    operator and its vectors."""
    entries = 4.0 * n * _factor_entries(n, eta, leaf, eps)
    return {"bytes": iterations * (entries * width + (56.0 + 64.0 * nrhs) * n ** 3),
            "flops": iterations * nrhs * (2.0 * entries + 40.0 * n ** 3)}


def work(case):
    kind = case["kind"]
    if kind == "operator":
        nodes = case["n"] ** 3
        fields = 3 if case["pde"] == "codi" else 1
        return {"bytes": 8.0 * nodes * (fields + 7 + 2 * case["nrhs"]),
                "flops": nodes * (30.0 + 13.0 * case["nrhs"])}
    parts = []
    if kind == "batch":
        for n in map(int, case["sizes"].split(",")):
            parts.append(_setup_work(n, case["eta"], case["leaf"], case["eps"], 4))
            parts.append(_solve_work(n, case["eta"], case["leaf"], case["eps"], 4, 1, 4))
    elif kind == "gradient":
        parts.append(_setup_work(case["n"], 2.0, 64, 1e-2, 4))
        parts.append(_solve_work(case["n"], 2.0, 64, 1e-2, 4, 1, 8))
    else:
        a = (case["n"], case["eta"], case["leaf"], case["eps"])
        if kind == "solve":
            parts.append(_setup_work(*a, _BYTES[case["prec"]]))
        parts.append(_solve_work(*a, _BYTES[case["prec"]], case.get("nrhs", 1), 4))
    return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}


# ------------------------------------------------------------------ exact values
def _shift(v, axis, step):
    """Neighbour values with zeros beyond the boundary."""
    out = torch.zeros_like(v)
    n = v.shape[axis]
    if step > 0:
        out.narrow(axis, 0, n - 1).copy_(v.narrow(axis, 1, n - 1))
    else:
        out.narrow(axis, 1, n - 1).copy_(v.narrow(axis, 0, n - 1))
    return out


# (axis, step) of the stencil's w, e, s, n, b, t in arrays indexed (z, y, x)
_DIRS = [(2, -1), (2, 1), (1, -1), (1, 1), (0, -1), (0, 1)]


def _face(kappa, axis, step):
    """Harmonic means of neighbouring nodes; the node's own value on the boundary."""
    other = kappa.clone()
    n = kappa.shape[axis]
    if step > 0:
        other.narrow(axis, 0, n - 1).copy_(kappa.narrow(axis, 1, n - 1))
    else:
        other.narrow(axis, 1, n - 1).copy_(kappa.narrow(axis, 0, n - 1))
    return 2.0 * kappa * other / (kappa + other)


def _stencil(pde, n, field):
    """The seven coefficient arrays c, w, e, s, n, b, t, each (z, y, x)."""
    h2 = float((n + 1) ** 2)
    if pde == "poisson":
        kappa = field.reshape(n, n, n)
        offs = [-h2 * _face(kappa, a, s) for a, s in _DIRS]
        centre = -sum(offs)
    elif pde == "codi":
        beta = field.reshape(3, n, n, n)
        h1 = float(n + 1)
        offs = []
        centre = torch.full((n, n, n), 6.0 * h2, dtype=torch.float64, device=field.device)
        for d in range(3):
            plus, minus = beta[d].clamp_min(0.0), beta[d].clamp_max(0.0)
            offs += [-h2 - h1 * plus, -h2 + h1 * minus]
            centre = centre + h1 * (plus - minus)
    else:
        offs = [torch.full((n, n, n), -h2, dtype=torch.float64, device=field.device)] * 6
        centre = 6.0 * h2 - field.reshape(n, n, n)
    return [centre] + offs


def _inside(st):
    """The seven arrays with the coefficients that point outside set to zero."""
    out = [st[0]]
    for (axis, step), o in zip(_DIRS, st[1:]):
        o = o.clone()
        n = o.shape[axis]
        o.narrow(axis, n - 1 if step > 0 else 0, 1).zero_()
        out.append(o)
    return out


def _mul(st, x):
    y = st[0] * x
    for (axis, step), o in zip(_DIRS, st[1:]):
        y = y + o * _shift(x, axis, step)
    return y


def _sines(n):
    i = torch.arange(1, n + 1, dtype=torch.float64, device=_DEV)
    return math.sqrt(2.0 / (n + 1)) * torch.sin(math.pi / (n + 1) * i[:, None] * i[None, :])


def _separable(n, scale, shift):
    """x -> (scale (-Lap_h) - diag_x(shift))^-1 x in 64 bits: sine transforms along
    z and y, eigenvectors of the 1D operator along x."""
    h2 = float((n + 1) ** 2)
    one = 2.0 * torch.eye(n, dtype=torch.float64, device=_DEV)
    one -= torch.diag(torch.ones(n - 1, dtype=torch.float64, device=_DEV), 1)
    one -= torch.diag(torch.ones(n - 1, dtype=torch.float64, device=_DEV), -1)
    s = _sines(n)
    i = torch.arange(1, n + 1, dtype=torch.float64, device=_DEV)
    lam = scale * h2 * (2.0 - 2.0 * torch.cos(math.pi * i / (n + 1)))
    mu, q = torch.linalg.eigh(scale * h2 * one - torch.diag(shift))
    den = lam[:, None, None] + lam[None, :, None] + mu[None, None, :]

    def solve(x):
        x = torch.einsum("ab,bcd->acd", s, x)
        x = torch.einsum("ab,cbd->cad", s, x)
        x = torch.matmul(x, q) / den
        x = torch.matmul(x, q.T)
        x = torch.einsum("ab,cbd->cad", s, x)
        return torch.einsum("ab,bcd->acd", s, x)

    return solve


def _bicgstab(mul, pre, b, rtol, maxit):
    x = torch.zeros_like(b)
    r = b.clone()
    r0 = r.clone()
    rho = alpha = omega = 1.0
    v = torch.zeros_like(b)
    p = torch.zeros_like(b)
    goal = rtol * float(b.norm())
    for _ in range(maxit):
        rho_new = float((r0 * r).sum())
        if rho_new == 0.0 or omega == 0.0:
            break
        beta = (rho_new / rho) * (alpha / omega)
        rho = rho_new
        p = r + beta * (p - omega * v)
        ph = pre(p)
        v = mul(ph)
        alpha = rho / float((r0 * v).sum())
        s = r - alpha * v
        sh = pre(s)
        t = mul(sh)
        tt = float((t * t).sum())
        omega = float((t * s).sum()) / tt if tt else 0.0
        x = x + alpha * ph + omega * sh
        r = s - omega * t
        if float(r.norm()) <= goal:
            break
    return x


def _inverse(pde, n, st, field, b):
    """A^-1 b in 64 bits: the separable operator directly, the others by a
    preconditioned iteration with refinement of the true residual."""
    zero = torch.zeros(n, dtype=torch.float64, device=_DEV)
    b = b.reshape(n, n, n)
    if pde == "helmholtz":
        pre = _separable(n, 1.0, field.reshape(n, n, n)[0, 0])
        x = pre(b)
        for _ in range(3):
            x = x + pre(b - _mul(st, x))
        return x.reshape(-1)
    if pde == "codi":
        pre = _separable(n, 1.0, zero)
    else:
        # symmetric scaling by sqrt(kappa) around the constant-coefficient inverse
        w = field.reshape(n, n, n).rsqrt()
        lap = _separable(n, 1.0, zero)

        def pre(x):
            return w * lap(w * x)
    x = torch.zeros_like(b)
    best, at = None, math.inf
    for _ in range(6):
        r = b - _mul(st, x)
        size = float(r.norm() / b.norm())
        if size < at:
            best, at = x, size
        elif best is not None:
            break
        if size < 1e-15:
            break
        x = x + _bicgstab(lambda v: _mul(st, v), pre, r, 1e-8, 400)
    return best.reshape(-1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        out = []
        for n, (kappa, f) in zip(map(int, case["sizes"].split(",")), _fields(case, seed)):
            out.append(_inverse("poisson", n, _inside(_stencil("poisson", n, kappa)), kappa, f))
        return out
    field, f = _fields(case, seed)
    n = case["n"]
    pde = case.get("pde", "poisson")
    st = _stencil(pde, n, field)
    if kind == "operator":
        st = _inside(st)
        y = [_mul(st, v.reshape(n, n, n)).reshape(-1) for v in f.reshape(case["nrhs"], -1)]
        return {"coef": torch.cat([o.reshape(-1) for o in st]), "y": torch.cat(y)}
    if kind == "gradient":
        g = _uniform(_gen(seed + 1000003), -1.0, 1.0, n ** 3)
        u = _inverse(pde, n, _inside(st), field, f)
        lam = _inverse(pde, n, _inside(st), field, g)
        kappa = field.clone().requires_grad_(True)
        y = _mul(_stencil(pde, n, kappa), u.reshape(n, n, n))
        (grad,) = torch.autograd.grad(-(lam.reshape(n, n, n) * y).sum(), kappa)
        return {"u": u, "kappa": grad, "f": lam}
    inside = _inside(st)
    return torch.cat([_inverse(pde, n, inside, field, v)
                      for v in f.reshape(case.get("nrhs", 1), -1)])

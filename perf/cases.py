"""Timing cases of the library's public entry points.

Each case is one call (or one burst of served requests) as a user's program
makes it: eigenvalue counts of a CSR matrix or of a finite-difference
Hamiltonian through ``Context.count_slices`` or ``evc_count_slices_async``,
requests through the server, and the allocation-free quadrature.  Sizes and
options are those of ``workloads.py``, the tests and the benchmark: the paper's
Laplace problem, FD Hamiltonians with Gaussian wells (identity, Jacobi and
Chebyshev preconditioners), and power-law sparse matrices, in both precisions.

  listed()   the cases; draw(rng) one more of the same ranges
  prepare()  inputs, context and preconditioner (what a program keeps)
  run()      one call; its outputs
  work()     bytes and operations that the call cannot do without
  exact()    the same outputs from plain torch in float64
"""
import ctypes
import math

import numpy as np
import torch

from paper_1602_02306_gb300 import evc
from paper_1602_02306_gb300 import inputs as I

H = 0.3            # grid spacing of the FD Hamiltonians
EPS = 1e-3         # Jacobi: M = diag((|a_ii - tau| + EPS)^(-1/2))
DEGREE, CHEB_C = 8, 1.0

PRECISION = {"fp64": evc.EVC_FP64, "mixed": evc.EVC_MIXED}
PRECOND = {"identity": (evc.EVC_PREC_IDENTITY, 0.0, 0.0),
           "jacobi": (evc.EVC_PREC_JACOBI, EPS, 0.0),
           "cheb": (evc.EVC_PREC_CHEB_KINETIC, float(DEGREE), CHEB_C)}


def _count(name, matrix, size, order, precision, precond, lo, hi, shifts, probes, steps, **kw):
    case = {"name": name, "kind": "count", "matrix": matrix, "size": size, "order": order,
            "precision": precision, "precond": precond, "lo": lo, "hi": hi, "shifts": shifts,
            "probes": probes, "steps": steps, "tol": 0.0, "min_steps": 3, "method": "lanczos",
            "rule": "gauss", "tiles": "default", "results": "host"}
    case.update(kw)
    return case


def listed():
    return [
        # quadratures of tridiagonals another program has on the device: the
        # smallest call, one launch without any allocation
        {"name": "quadrature 64 x k=40", "kind": "quad", "columns": 64, "k": 40},
        # the plain FP64 problem: n = 1024, everything is launches and latency
        _count("laplace 32^2 fp64", "laplace", 32, 0, "fp64", "jacobi", 1.0, 2.0, 2, 16, 40),
        # the paper's Table 1 problem: many steps on a small matrix, one shift, ragged probes
        _count("laplace 127^2 k=134", "laplace", 127, 0, "mixed", "jacobi", 3000.0, 3000.0, 1, 50, 134),
        # a small interactive count: shifts share a Lanczos run, stop by tolerance,
        # results stay on the device
        _count("fd 32^3 shared, stop", "fd", 32, 2, "mixed", "identity", -4.0, -1.0, 4, 64, 30,
               tol=0.25, min_steps=10, results="device"),
        # requests that arrive together at the server, on matrices of three sizes
        {"name": "server burst", "kind": "serve", "size": 40, "requests": 12, "probes": 32, "steps": 30},
        # the Arnoldi-type estimator
        _count("fd 40^3 arnoldi", "fd", 40, 2, "mixed", "cheb", -3.0, 0.5, 2, 32, 24, method="arnoldi"),
        # full FP64 on a grid with the averaged Gauss rule, library defaults
        _count("fd 40^3 fp64 averaged", "fd", 40, 2, "fp64", "cheb", -4.0, 0.5, 2, 32, 30, rule="averaged"),
        # full FP64 on a generic sparse matrix; probes that do not fill their chunks
        _count("sparse 200k fp64", "powerlaw", 200003, 0, "fp64", "jacobi", -0.5, 0.5, 2, 40, 40),
        # the DFT-like count: Chebyshev preconditioner, tuned tiles
        _count("fd 64^3 chebyshev", "fd", 64, 2, "mixed", "cheb", -4.28, 0.51, 2, 64, 30, tiles="tuned"),
        # the T^-1-inner-product process
        _count("sparse 600k tinv", "powerlaw", 600000, 0, "mixed", "jacobi", -0.5, 0.5, 2, 64, 30,
               method="tinv", tiles="tuned"),
        # spectrum slicing with the 13-point stencil and early stop
        _count("fd 96^3 slicing", "fd", 96, 4, "mixed", "cheb", -2.2, 5.2, 4, 64, 30, tol=0.25,
               min_steps=10, tiles="tuned"),
        # the large generic sparse count
        _count("sparse 2M", "powerlaw", 2000000, 0, "mixed", "jacobi", -0.5, 0.5, 2, 64, 30, tiles="tuned"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    which = rng.choice(["quad", "laplace", "laplace", "fd", "fd", "fd", "sparse", "sparse", "arnoldi",
                        "slicing", "serve"])
    results = rng.choice(["host", "device"])
    if which == "quad":
        k = _log_int(rng, 8, 200)
        return {"kind": "quad", "columns": _log_int(rng, 16, min(4096, 262144 // k)), "k": k}
    if which == "serve":
        return {"kind": "serve", "size": rng.randrange(24, 65), "requests": rng.randrange(4, 17),
                "probes": rng.choice([32, 64]), "steps": 30}
    if which == "laplace":
        N = _log_int(rng, 16, 300)
        k = _log_int(rng, 20, 60)
        lo = 8.0 * rng.uniform(0.1, 0.3)
        case = _count("", "laplace", N, 0, rng.choice(["fp64", "mixed"]), "jacobi", lo, lo + 1.0,
                      rng.choice([1, 2]), rng.randrange(8, 65), k, rule=rng.choice(["gauss", "averaged"]))
    elif which == "fd":
        N = _log_int(rng, 16, 72)
        precision = rng.choice(["fp64", "mixed", "mixed"])
        precond = rng.choice(["identity", "jacobi", "cheb", "cheb"])
        case = _count("", "fd", N, rng.choice([2, 2, 4]), precision, precond, -4.0, rng.uniform(-1.0, 0.5),
                      rng.choice([2, 2, 3]), rng.randrange(16, 33 if precision == "fp64" else 65),
                      rng.randrange(12, 31), tiles=rng.choice(["default", "tuned"]))
    elif which == "sparse":
        precision = rng.choice(["fp64", "mixed", "mixed"])
        n = _log_int(rng, 5000, 200000 if precision == "fp64" else 1500000)
        case = _count("", "powerlaw", n, 0, precision, rng.choice(["jacobi", "jacobi", "identity"]),
                      -0.5, 0.5, rng.choice([1, 2, 2]), rng.randrange(16, 65), rng.randrange(12, 31),
                      tiles=rng.choice(["default", "tuned"]))
        if case["precond"] == "jacobi" and rng.random() < 0.3:
            case["method"] = "tinv"
    elif which == "arnoldi":
        case = _count("", "fd", _log_int(rng, 16, 48), 2, rng.choice(["fp64", "mixed"]),
                      rng.choice(["jacobi", "cheb"]), -3.0, 0.5, 2, rng.randrange(16, 33),
                      rng.randrange(12, 31), method="arnoldi")
    else:
        S = rng.randrange(2, 6)
        case = _count("", "fd", rng.choice([48, 56, 64, 72, 80]), rng.choice([2, 4]), "mixed", "cheb",
                      -2.2, 5.2, S, rng.choice([32, 48, 64]), 30, tol=0.25, min_steps=10, tiles="tuned")
    case["results"] = results
    del case["name"]
    return case


# ------------------------------------------------------------------ inputs

def _shifts(case):
    return [float(x) for x in np.linspace(case["lo"], case["hi"], case["shifts"])] \
        if case["shifts"] > 1 else [float(case["lo"])]


def _potential(N, seed):
    return I.gaussian_wells(N, H, nwells=32, seed=seed % (1 << 30) + 1)


def _powerlaw(n, seed):
    """A = B + B^T with Pareto out-degrees, uniform columns, N(0,1) values and
    a U(-5, 5) diagonal (the recipe of inputs.powerlaw_symmetric), built on the
    GPU; entries drawn twice stay stored twice."""
    g = torch.Generator(device="cuda").manual_seed(seed % (1 << 30) + 2)
    dev = {"device": "cuda", "generator": g}
    raw = (1.0 - torch.rand(n, dtype=torch.float64, **dev)).pow(-1.0 / 1.2).clamp(max=2000.0)
    deg = (raw * (14.5 / raw.mean())).round().clamp(max=2000.0).long()
    r = torch.repeat_interleave(torch.arange(n, device="cuda"), deg)
    c = torch.randint(0, n, (r.numel(),), **dev)
    v = torch.randn(r.numel(), dtype=torch.float64, **dev)
    keep = r != c
    r, c, v = r[keep], c[keep], v[keep]
    d = torch.rand(n, dtype=torch.float64, **dev) * 10.0 - 5.0
    i = torch.arange(n, device="cuda")
    key, order = torch.sort(torch.cat([r * n + c, c * n + r, i * n + i]), stable=True)
    val = torch.cat([v, v, d])[order]
    rows = torch.div(key, n, rounding_mode="floor")
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    row_ptr[1:] = torch.cumsum(torch.bincount(rows, minlength=n), 0)
    return row_ptr, (key - rows * n).int(), val


def _laplace(N):
    # h = 1/(N + 1) scaled by 1/h^2 for the paper's problem (tau = 3000 on 127^2)
    return I.laplace2d_dirichlet(N, scale=float((N + 1) ** 2) if N == 127 else 1.0)


def _context(case, seed):
    """The context and what has to stay alive with it."""
    precision = PRECISION[case["precision"]]
    keep = None
    if case["matrix"] == "fd":
        ctx = evc.Context.stencil(case["size"], H, case["order"], _potential(case["size"], seed),
                                  precision=precision)
    elif case["matrix"] == "laplace":
        ctx = evc.Context.csr(_laplace(case["size"]), precision=precision)
    else:
        keep = _powerlaw(case["size"], seed)
        torch.cuda.synchronize()
        ctx = evc.Context(evc.evc_create_csr(*keep, precision=precision, on_device=True))
    ctx.set_precond(*PRECOND[case["precond"]])
    ctx.set_option(evc.EVC_OPT_MIN_STEPS, case["min_steps"])
    if case["rule"] == "averaged":
        ctx.set_option(evc.EVC_OPT_QUADRATURE, evc.EVC_QUAD_GA)
    if case["method"] == "arnoldi":
        ctx.set_option(evc.EVC_OPT_METHOD, evc.EVC_METHOD_ARNOLDI)
    if case["method"] == "tinv":
        ctx.set_option(evc.EVC_OPT_TINV_LANCZOS, 1)
    if case["tiles"] == "tuned":
        # the shapes that the autotuner settles on for these problems
        if case["matrix"] != "fd":
            ctx.set_option(evc.EVC_OPT_CSR_THREADS, 128)
        elif case["order"] == 2:
            ctx.set_option(evc.EVC_OPT_STENCIL_PATCH, 3)
            ctx.set_option(evc.EVC_OPT_STENCIL_ZB, 32)
            ctx.set_option(evc.EVC_OPT_STENCIL_GROUPS, 4)
        else:
            ctx.set_option(evc.EVC_OPT_STENCIL_PATCH, 2)
            ctx.set_option(evc.EVC_OPT_STENCIL_ZB, 64)
    return ctx, keep


class _Served:
    """Three resident Hamiltonians, a server over them and a burst of requests."""

    def __init__(self, case, seed):
        self.ctxs, self.requests = [], _requests(case, seed)
        for N in _served_sizes(case):
            ctx = evc.Context.stencil(N, H, 2, _potential(N, seed), precision=evc.EVC_MIXED)
            ctx.set_option(evc.EVC_OPT_MIN_STEPS, 10)
            self.ctxs.append(ctx)
        self.srv = evc.evc_server_create(16 << 30, slots=2, max_batch=16)
        self.ids = [evc.evc_server_add_matrix(self.srv, c.h) for c in self.ctxs]

    def __del__(self):
        evc.evc_server_destroy(self.srv)
        for c in self.ctxs:
            c.close()


def _served_sizes(case):
    return [case["size"], (case["size"] * 5) // 4, (case["size"] * 3) // 2]


def _requests(case, seed):
    rng = np.random.default_rng(seed)
    out = []
    for q in range(case["requests"]):
        a, b = np.sort(rng.uniform(-4.0, 0.0, size=2))
        out.append({"matrix": int(rng.integers(0, 3)), "xi": float(a), "eta": float(b) + 0.05,
                    "tol": float(rng.choice([0.25, 0.5]))})
    return out


def prepare(case, seed):
    if case["kind"] == "quad":
        # Lanczos coefficients of a spectrum on [-2, 2]: alpha around 0, beta around 1
        g = torch.Generator(device="cuda").manual_seed(seed % (1 << 30))
        k, nc = case["k"], case["columns"]
        alpha = torch.randn(k, nc, dtype=torch.float64, device="cuda", generator=g) * 0.3
        beta = 0.7 + 0.6 * torch.rand(k + 1, nc, dtype=torch.float64, device="cuda", generator=g)
        return {"case": case, "alpha": alpha, "beta": beta,
                "quad": torch.empty(nc, dtype=torch.float64, device="cuda"),
                "status": torch.empty(1, dtype=torch.int32, device="cuda")}
    if case["kind"] == "serve":
        return {"case": case, "served": _Served(case, seed)}
    ctx, keep = _context(case, seed)
    state = {"case": case, "ctx": ctx, "keep": keep, "shifts": _shifts(case), "seed": seed}
    if case["results"] == "device":
        S, m = case["shifts"], case["probes"]
        state["n_below"] = torch.empty(S, dtype=torch.float64, device="cuda")
        state["quad"] = torch.empty(S, m, dtype=torch.float64, device="cuda")
        state["steps"] = torch.empty(S, dtype=torch.int32, device="cuda")
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "quad":
        rc, msg = evc.evc_gauss_quadrature_static(
            state["alpha"].data_ptr(), state["beta"].data_ptr(), None, case["k"], case["columns"], 1.0,
            state["quad"].data_ptr(), state["status"].data_ptr(), None)
        if rc != evc.EVC_OK:
            raise RuntimeError(msg)
        return {"quad": state["quad"], "status": state["status"]}
    if case["kind"] == "serve":
        s = state["served"]
        quads = [np.zeros(2 * case["probes"]) for _ in s.requests]
        tickets = [evc.evc_server_submit(s.srv, s.ids[q["matrix"]], q["xi"], q["eta"], case["probes"],
                                         case["steps"], q["tol"], 3, b)
                   for q, b in zip(s.requests, quads)]
        results = []
        for t in tickets:
            rc, r = evc.evc_server_wait(s.srv, t)
            if rc != evc.EVC_OK:
                raise evc.EvcError(rc, "served request failed")
            results.append(r)
        return {"n_below": np.array([r["n_below"] for r in results]), "quad": np.stack(quads),
                "steps": np.array([r["steps"] for r in results])}
    ctx, m, k = state["ctx"], case["probes"], case["steps"]
    if case["results"] == "device":
        ctx.reserve(case["shifts"], m, k)
        evc.evc_count_slices_async(ctx.h, state["shifts"], m, k, case["tol"], state["seed"],
                                   ctypes.c_void_p(state["n_below"].data_ptr()),
                                   ctypes.c_void_p(state["quad"].data_ptr()),
                                   ctypes.c_void_p(state["steps"].data_ptr()))
        return {"n_below": state["n_below"], "quad": state["quad"], "steps": state["steps"]}
    L, quad, steps = ctx.count_slices(state["shifts"], m, k, tol=case["tol"], seed=state["seed"])
    return {"n_below": L, "quad": quad, "steps": steps}


# -------------------------------------------------------------------- work

def _eig_flops(k):
    return 30.0 * k * k          # QR with the first components: about 1.7 k sweeps of k/2 rotations


def _run_work(n, nnz, columns, quads, k, size, precond, order, fd):
    """k Lanczos steps on `columns` vectors of n elements of `size` bytes.  A
    step reads the basis once for the projections and once to subtract them
    (the coefficients need the whole of the first sweep), and the operator
    reads its operand and q_(i-1) and writes one vector; the matrix or the
    potential is read once."""
    vec = float(n) * columns * size
    steps = k * 3.0 + (k * (k + 1) / 2.0 + k) * 2.0
    mat = n * size if fd else nnz * (size + 4.0) + 8.0 * n
    points = (13.0 if order == 4 else 7.0) * n if fd else float(nnz)
    applies = 1 + 2 * DEGREE if precond == "cheb" else 1
    flops = n * columns * (2.0 * points / n * applies * k + 3.0 * k * (k + 1)) + quads * _eig_flops(k)
    return {"bytes": vec * steps + k * mat, "flops": flops}


def work(case):
    if case["kind"] == "quad":
        k, nc = case["k"], case["columns"]
        return {"bytes": 8.0 * nc * (2 * k + 1) + 8.0 * nc, "flops": nc * _eig_flops(k)}
    if case["kind"] == "serve":
        # every request at its first possible stop; one Lanczos run per matrix
        # serves all of its requests
        total = {"bytes": 0.0, "flops": 0.0}
        for N in _served_sizes(case):
            w = _run_work(N ** 3, 0, case["probes"], case["probes"], 10, 4, "identity", 2, True)
            total = {key: total[key] + w[key] for key in total}
        return total
    size = 8 if case["precision"] == "fp64" else 4
    fd = case["matrix"] == "fd"
    n = case["size"] ** 3 if fd else case["size"] ** 2 if case["matrix"] == "laplace" else case["size"]
    nnz = 0 if fd else 5 * n if case["matrix"] == "laplace" else 30 * n
    shared = case["precond"] == "identity" and case["method"] == "lanczos"
    columns = case["probes"] * (1 if shared else case["shifts"])
    k = case["min_steps"] + 2 if case["tol"] > 0 else case["steps"]
    k = min(k, n)
    return _run_work(n, nnz, columns, case["probes"] * case["shifts"], k, size, case["precond"],
                     case["order"], fd)


# ------------------------------------------------------------------- exact

def _mix(z):
    def srl(x, s):
        return (x >> s) & ((1 << (64 - s)) - 1)

    def signed(x):
        return x - (1 << 64) if x >= 1 << 63 else x
    z = (z ^ srl(z, 30)) * signed(0xbf58476d1ce4e5b9)
    z = (z ^ srl(z, 27)) * signed(0x94d049bb133111eb)
    return z ^ srl(z, 31)


def _probes(n, m, seed):
    i = torch.arange(n, dtype=torch.int64, device="cuda")[:, None]
    j = torch.arange(m, dtype=torch.int64, device="cuda")[None, :]
    x = _mix(seed ^ _mix((j << 32) | i))
    return torch.where(x < 0, -1.0, 1.0).double()


def _laplacian(order):
    """Weights of -1/2 Lap_h along one axis at offsets 0, 1, 2 (times 1/h^2)."""
    return (1.0, -0.5, 0.0) if order == 2 else (30.0 / 24.0, -16.0 / 24.0, 1.0 / 24.0)


def _kinetic(x, N, order):
    w0, w1, w2 = _laplacian(order)
    g = x.view(N, N, N, -1)
    y = 3.0 * w0 * g
    for axis in range(3):
        y += w1 * (torch.roll(g, 1, axis) + torch.roll(g, -1, axis))
        if order == 4:
            y += w2 * (torch.roll(g, 2, axis) + torch.roll(g, -2, axis))
    return (y / (H * H)).view(N ** 3, -1)


def _cheb_apply(x, N, order):
    """p_d(K) x, K = -1/2 Lap_h + c, p_d interpolating x^(-1/2) at the d + 1
    Chebyshev points of [c, c + 6/h^2] (7-point) or [c, c + 8/h^2] (13-point)."""
    a, b = CHEB_C, CHEB_C + (6.0 if order == 2 else 8.0) / (H * H)
    t = np.cos(np.pi * (2 * np.arange(DEGREE + 1) + 1) / (2.0 * (DEGREE + 1)))
    f = 1.0 / np.sqrt(0.5 * (a + b) + 0.5 * (b - a) * t)
    c = np.polynomial.chebyshev.chebfit(t, f, DEGREE)
    b1 = b2 = None
    for j in range(DEGREE, -1, -1):
        y = c[j] * x
        if b1 is not None:
            k = _kinetic(b1, N, order) + CHEB_C * b1
            y += (1.0 if j == 0 else 2.0) * (2.0 * k - (a + b) * b1) / (b - a)
        if b2 is not None:
            y -= b2
        b1, b2 = y, b1
    return b1


class _Operator:
    """C = M (A - tau) M (Lanczos) or T (A - tau), T = M^2 (Arnoldi), applied to
    the columns of all shifts at once; tau holds one shift per column."""

    def __init__(self, case, seed, tau):
        self.case, self.tau = case, tau
        N = case["size"]
        if case["matrix"] == "fd":
            self.V = torch.from_numpy(_potential(N, seed)).cuda()[:, None]
            diag = self.V + 3.0 * _laplacian(case["order"])[0] / (H * H)
        else:
            if case["matrix"] == "laplace":
                rp, ci, va = (torch.from_numpy(x).cuda() for x in _laplace(N))
            else:
                rp, ci, va = _powerlaw(N, seed)
            n = rp.numel() - 1
            rows = torch.repeat_interleave(torch.arange(n, device="cuda"), rp[1:] - rp[:-1])
            self.A = torch.sparse_csr_tensor(rp, ci.long(), va, size=(n, n))
            on = rows == ci
            diag = torch.zeros(n, dtype=torch.float64, device="cuda")
            diag[rows[on]] = va[on]          # one stored diagonal entry per row
            diag = diag[:, None]
        self.n = diag.shape[0]
        self.m2 = None
        if case["precond"] == "jacobi":
            self.diag = diag

    def matvec(self, x):
        if self.case["matrix"] == "fd":
            return _kinetic(x, self.case["size"], self.case["order"]) + self.V * x
        return self.A @ x

    def scale(self, x, power):
        """M^power x of the preconditioner, power 1 or 2."""
        kind = self.case["precond"]
        if kind == "identity":
            return x
        if kind == "jacobi":
            t = 1.0 / ((self.diag - self.tau).abs_().add_(EPS))
            return x * (t if power == 2 else t.sqrt_())
        for _ in range(power):
            x = _cheb_apply(x, self.case["size"], self.case["order"])
        return x

    def __call__(self, x):
        if self.case["method"] == "arnoldi":
            y = self.matvec(x)
            return self.scale(y.sub_(self.tau * x), 2)
        x = self.scale(x, 1)
        y = self.matvec(x)
        return self.scale(y.sub_(self.tau * x), 1)


def _rule(alpha, beta, averaged):
    """Eigenvalues and squared first components of J_k (columns first), or of
    the extended matrix of the generalized averaged Gauss rule."""
    k = alpha.shape[1]
    off = beta[:, 1:k]
    if averaged and k > 1:
        alpha = torch.cat([alpha, alpha[:, :-1].flip(1)], 1)
        off = torch.cat([off, beta[:, k:k + 1], off[:, :-1].flip(1)], 1)
    J = torch.diag_embed(alpha)
    if off.shape[1]:
        J = J + torch.diag_embed(off, 1) + torch.diag_embed(off, -1)
    theta, Z = torch.linalg.eigh(J.cpu())
    return theta.cuda(), (Z[:, 0, :] ** 2).cuda()


def _arnoldi_quad(Hk):
    """Re e_1^T h(H) e_1 per column from the eigen-decomposition of H."""
    w, Z = np.linalg.eig(Hk)
    return np.real(Z[:, 0, :] * np.linalg.inv(Z)[:, :, 0] * (w.real < 0)).sum(1)


def _lanczos(case, seed, op, columns, averaged, quadratures):
    """k steps with full reorthogonalisation (two sweeps), calling quadratures(i,
    alpha, beta, H) after each step; stops when it returns True."""
    n, k = op.n, min(case["steps"], op.n)
    v = _probes(n, case["probes"], case.get("probe_seed", seed))
    q = (v / math.sqrt(n)).repeat(1, columns // case["probes"])
    del v
    arnoldi = case["method"] == "arnoldi"
    Q = torch.empty(k + 1, n, columns, dtype=torch.float64, device="cuda")
    Q[0] = q
    alpha = torch.zeros(columns, k, dtype=torch.float64, device="cuda")
    beta = torch.zeros(columns, k + 1, dtype=torch.float64, device="cuda")
    Hk = torch.zeros(columns, k + 1, k, dtype=torch.float64, device="cuda")
    for i in range(1, k + 1):
        w = op(Q[i - 1])
        if not arnoldi and i > 1:
            w -= beta[:, i - 1] * Q[i - 2]
        for sweep in range(2):
            for j in range(i):
                h = (Q[j] * w).sum(0)
                w.addcmul_(Q[j], h[None, :], value=-1.0)
                Hk[:, j, i - 1] += h
                if j == i - 1:
                    alpha[:, i - 1] += h
        nrm = w.norm(dim=0)
        beta[:, i] = nrm
        Hk[:, i, i - 1] = nrm
        Q[i] = w / nrm
        if quadratures(i, alpha[:, :i], beta[:, :i + 1], Hk[:, :i, :i]):
            break


def _exact_count(case, seed, shifts, tols):
    """Quadratures, means and stop steps of every shift (the rule: the first
    step i >= max(3, min_steps) at which the mean moved by at most tol twice)."""
    S, m = len(shifts), case["probes"]
    shared = case["precond"] == "identity" and case["method"] != "arnoldi"
    columns = m if shared else S * m
    tau = torch.zeros(m, dtype=torch.float64, device="cuda") if shared else \
        torch.tensor(shifts, dtype=torch.float64, device="cuda").repeat_interleave(m)
    op = _Operator(case, seed, tau[None, :])
    k = min(case["steps"], op.n)
    means = [[] for _ in range(S)]
    quad, steps = np.zeros((S, m)), np.zeros(S, dtype=np.int32)

    def quadratures(i, alpha, beta, Hk):
        if max(tols) <= 0.0 and i < k:
            return False
        if case["method"] == "arnoldi":
            rows = _arnoldi_quad(Hk.cpu().numpy()).reshape(S, m) * op.n
        else:
            theta, z2 = _rule(alpha, beta, case["rule"] == "averaged")
            if shared:
                rows = np.stack([(z2 * (theta < s)).sum(1).cpu().numpy() for s in shifts]) * op.n
            else:
                rows = (z2 * (theta < 0.0)).sum(1).cpu().numpy().reshape(S, m) * op.n
        for s in range(S):
            if steps[s]:
                continue
            L = means[s]
            L.append(float(rows[s].mean()))
            stop = i == k or (tols[s] > 0.0 and i >= max(3, case["min_steps"]) and
                              abs(L[-1] - L[-2]) <= tols[s] and abs(L[-2] - L[-3]) <= tols[s])
            if stop:
                quad[s], steps[s] = rows[s], i
        return bool((steps > 0).all())

    _lanczos(case, seed, op, columns, case["rule"] == "averaged", quadratures)
    return quad.mean(1), quad, steps


def exact(case, seed):
    if case["kind"] == "quad":
        s = prepare(case, seed)
        theta, z2 = _rule(s["alpha"].T.contiguous(), s["beta"].T.contiguous(), False)
        return {"quad": (z2 * (theta < 0.0)).sum(1), "status": None}
    if case["kind"] == "serve":
        L, quad, steps = [], [], []
        sizes = _served_sizes(case)
        for q in _requests(case, seed):
            one = {"kind": "count", "matrix": "fd", "size": sizes[q["matrix"]], "order": 2,
                   "precond": "identity", "probes": case["probes"], "steps": case["steps"],
                   "min_steps": 10, "method": "lanczos", "rule": "gauss", "probe_seed": 3}
            l1, q1, s1 = _exact_count(one, seed, [q["xi"], q["eta"]], [q["tol"], q["tol"]])
            L.append(l1)
            quad.append(q1.reshape(-1))
            steps.append(s1)
        return {"n_below": np.stack(L), "quad": np.stack(quad), "steps": None}
    shifts = _shifts(case)
    L, quad, _ = _exact_count(case, seed, shifts, [case["tol"]] * len(shifts))
    return {"n_below": L, "quad": quad, "steps": None}

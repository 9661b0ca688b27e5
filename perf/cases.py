"""The work users of this library have it do, as measurable cases.

A case is one call path of the public binding (`paper_2406_00952_gb300`): a whole control solve from
samples of the target g and the source f to the state y and the adjoint p (assemble_rhs -> solve ->
recover), the same solve through host buffers, a batch of uneven solves, and the single steps a
caller can take alone (the preconditioner apply in FP64, the all-at-once product, one Lanczos step).
Sizes, parameters and data are those of the repository's configurations, tests and benchmark.
"""
import math

import numpy as np
import torch

import paper_2406_00952_gb300 as pcb

PI = math.pi

# Grids the transforms support: N + 1 = 2^a 3^b (Dirichlet), N - 1 = 2^a 3^b (Neumann).
DIRICHLET = (15, 23, 31, 47, 63, 95, 127, 191, 255, 383, 511)
NEUMANN = (17, 33, 49, 65, 97, 129, 193, 257)
MULTIGRID = (15, 31, 63, 127, 255)
STEPS = (16, 32, 64, 128, 256, 512)


def _case(op, N, n, **kw):
    c = {"op": op, "N": N, "n": n, "theta": 1.0, "gamma": 1e-2, "zeta": PI, "bc": "dirichlet", "a": 1.0,
         "precision": "mixed", "tol": 1e-10, "variable_a": False, "kind": "abs_ps", "count": 1, "pick": 0}
    c.update(kw)
    return c


def listed():
    return [
        # the smallest problem of the configurations: launches and latency of an FP64 solve
        dict(_case("solve", 15, 16, precision="fp64"), name="fp64 minres 15x16"),
        # a small Crank-Nicolson solve (GMRES with P_S), as an interactive user or a test runs it
        dict(_case("solve", 63, 64, theta=0.5, gamma=1e-3), name="mixed gmres cn 63x64"),
        # an ordinary FP64 solve on a grid that is no power of two (N + 1 = 192)
        dict(_case("solve", 191, 128, gamma=1e-3, precision="fp64"), name="fp64 minres 191x128"),
        # the same method at omega = i, the fastest choice of omega for this family
        dict(_case("solve", 255, 256, gamma=1e-6, zeta=PI / 2), name="mixed minres omega i 255x256"),
        # the benchmark's workload: the largest single instance, 2.7e8 unknowns
        dict(_case("solve", 511, 512, tol=1e-8), name="mixed minres 511x512"),
        # Example 3: homogeneous Neumann data, Crank-Nicolson, small diffusion
        dict(_case("solve", 257, 256, theta=0.5, bc="neumann", a=1e-3), name="mixed neumann gmres 257x256"),
        # variable coefficient: FGMRES with two V-cycles per shifted system
        dict(_case("solve", 255, 256, theta=0.5, gamma=1e-4, variable_a=True), name="mixed multigrid fgmres 255x256"),
        # end to end through page-locked host buffers
        dict(_case("host", 255, 256), name="mixed host solve 255x256"),
        # independent uneven requests in shared launches
        dict(_case("batch", 0, 0, count=12, pick=3), name="mixed uneven batch of 12"),
        # one P_S apply of an FP64 solver
        dict(_case("apply", 255, 256, theta=0.5, gamma=1e-4, precision="fp64", kind="ps"), name="fp64 apply ps 255x256"),
        # the operator product of a Crank-Nicolson residual
        dict(_case("product", 255, 256, theta=0.5, gamma=1e-4, precision="fp64"), name="fp64 product cn 255x256"),
        # one Lanczos step in the arithmetic of the mixed solver's inner iterations
        dict(_case("lanczos", 511, 256), name="mixed lanczos step 511x256"),
    ]


def draw(rng):
    op = rng.choice(("solve",) * 7 + ("host", "batch", "apply", "apply", "product", "lanczos"))
    gamma = 10.0 ** rng.uniform(-6.0, -1.0)
    if op == "batch":
        return _case("batch", 0, 0, count=rng.randint(4, 16), pick=rng.randrange(1 << 20), gamma=gamma)
    theta = rng.choice((1.0, 0.5))
    precision = rng.choice(("mixed", "mixed", "mixed", "fp64"))
    kw = dict(theta=theta, gamma=gamma, precision=precision)
    grids = DIRICHLET
    if op == "solve":
        route = rng.choice(("plain", "plain", "plain", "omega", "neumann", "multigrid"))
        if route == "omega":
            kw.update(theta=1.0, zeta=PI / 2)
        elif route == "neumann":
            grids = NEUMANN
            kw.update(theta=0.5, bc="neumann", a=1e-3)
        elif route == "multigrid":
            grids = MULTIGRID
            kw.update(theta=0.5, variable_a=True)
    elif op == "host":
        kw.update(theta=1.0, precision="mixed")
    elif op == "apply":
        kw.update(precision="fp64", kind="abs_ps" if theta == 1.0 else "ps", zeta=rng.choice((PI, PI, PI / 2)))
    elif op == "product":
        kw.update(precision="fp64")
    elif op == "lanczos":
        kw.update(theta=1.0, precision="mixed")
    # the largest mixed MINRES solves and single steps; restarted GMRES keeps 62 vectors, an FP64 or a
    # host-buffer solve of the largest size would take seconds
    if op != "solve":
        most = 3.5e7 if op == "host" else 1.4e8
    elif kw["precision"] == "fp64":
        most = 1.7e7
    else:
        most = 1.4e8 if kw["theta"] == 1.0 else 3.5e7
    while True:
        N, n = rng.choice(grids), rng.choice(STEPS)
        if 2.0 * N * N * n <= most:
            return _case(op, N, n, **kw)


# ------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------
def _members(case):
    """The instances of a batch: uneven grids and horizons, as the benchmark's batch draws them."""
    rng = np.random.Generator(np.random.PCG64(case["pick"]))
    out = []
    for _ in range(case["count"]):
        N, n = int(rng.choice((63, 127, 191, 255))), int(rng.choice((32, 64, 128, 256)))
        out.append(dict(case, op="solve", N=N, n=n, theta=float(rng.choice((1.0, 0.5))),
                        gamma=float(10.0 ** rng.uniform(-6.0, -1.0))))
    return out


def _axis(case):
    N = case["N"]
    if case["bc"] == "neumann":
        return torch.arange(N, dtype=torch.float64, device="cuda") / (N - 1)
    return torch.arange(1, N + 1, dtype=torch.float64, device="cuda") / (N + 1)


def _samples(case, seed):
    """g and f at the n + 1 time levels: a random sum of low modes decaying in time, and a smooth
    source that grows in time (cosines instead of sines on the Neumann grid)."""
    rng = np.random.Generator(np.random.PCG64(seed))
    x = _axis(case)
    wave = torch.cos if case["bc"] == "neumann" else torch.sin
    space = torch.zeros(case["N"], case["N"], dtype=torch.float64, device="cuda")
    for _ in range(8):
        i, j = (int(k) for k in rng.integers(1, 5, size=2))
        c = float(rng.standard_normal()) / (i * i + j * j)
        space += c * torch.outer(wave(PI * j * x), wave(PI * i * x))
    t = torch.arange(case["n"] + 1, dtype=torch.float64, device="cuda") / case["n"]
    g = torch.exp(-t)[:, None] * space.reshape(1, -1)
    f = (1.0 + 2.0 * PI * PI * t)[:, None] * torch.outer(wave(PI * x), wave(PI * x)).reshape(1, -1)
    return g.reshape(-1), f.reshape(-1)


def _edges(N):
    """a(x) = 1 + 0.5 sin(pi x1) sin(pi x2) at the cell-edge midpoints."""
    h = 1.0 / (N + 1)
    node, mid = h * np.arange(1, N + 1), h * (np.arange(N + 1) + 0.5)
    along = 1.0 + 0.5 * np.outer(np.sin(PI * node), np.sin(PI * mid))
    return np.concatenate([along.ravel(), np.ascontiguousarray(along.T).ravel()])


def _problem(case):
    return pcb.Problem(case["N"], case["n"], case["theta"], case["gamma"], zeta=case["zeta"],
                       a_edges=_edges(case["N"]) if case["variable_a"] else None, precision=case["precision"],
                       bc=case["bc"], a=case["a"])


def _operator(case):
    """The system a default solve works on: symmetric for MINRES, nonsymmetric for (F)GMRES."""
    return "A" if case["theta"] == 1.0 and case["bc"] == "dirichlet" and not case["variable_a"] else "Ahat"


def _vector(size, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(size, dtype=torch.float64, device="cuda", generator=gen)


BETA, OLDB = 0.37, 0.59


def prepare(case, seed):
    op = case["op"]
    if op == "batch":
        parts = [prepare(m, seed + 101 * k) for k, m in enumerate(_members(case))]
        return {"case": case, "parts": parts}
    state = {"case": case, "problem": _problem(case)}
    size = state["problem"].size
    if op == "solve":
        state["g"], state["f"] = _samples(case, seed)
    elif op == "host":
        g, f = _samples(case, seed)
        b = state["problem"].assemble_rhs(g, f, op=_operator(case))
        state["b"] = b.cpu().pin_memory()
        state["x"] = torch.empty_like(state["b"]).pin_memory()
    else:
        state["x"], state["out"] = _vector(size, seed), torch.empty(size, dtype=torch.float64, device="cuda")
        if op == "lanczos":
            state["r"] = _vector(size, seed + 50021)
    return state


# ------------------------------------------------------------------------------------------
# the measured calls
# ------------------------------------------------------------------------------------------
def run(state):
    case, op = state["case"], state["case"]["op"]
    if op == "solve":
        problem = state["problem"]
        b = problem.assemble_rhs(state["g"], state["f"], op=_operator(case))
        x, _ = problem.solve(b, tol=case["tol"])
        y, p = problem.recover(x)
        return {"y": y, "p": p}
    if op == "host":
        x, _ = state["problem"].solve_host(state["b"], state["x"], tol=case["tol"])
        return {"x": x}
    if op == "batch":
        parts = state["parts"]
        bs = [s["problem"].assemble_rhs(s["g"], s["f"], op=_operator(s["case"])) for s in parts]
        xs, _ = pcb.batch_solve([s["problem"] for s in parts], bs, tol=case["tol"], restart=16)
        return [dict(zip("yp", s["problem"].recover(x))) for s, x in zip(parts, xs)]
    if op == "apply":
        return {"y": state["problem"].precond_apply(state["x"], out=state["out"], kind=case["kind"])}
    if op == "product":
        return {"y": state["problem"].matvec(state["x"], out=state["out"], op="A" if case["theta"] == 1.0 else "Ahat")}
    out, dot = state["problem"].lanczos_product(state["x"], BETA, state["r"], OLDB, out=state["out"])
    return {"out": out, "dot": dot}


def work(case):
    """A solve reads g and f and writes y and p once; the steps read and write 2 m n values each."""
    op = case["op"]
    if op == "batch":
        return {"bytes": sum(work(m)["bytes"] for m in _members(case)), "flops": 0.0}
    mn = float(case["N"]) ** 2 * case["n"]
    vectors = {"solve": 2, "host": 2, "apply": 2, "product": 2, "lanczos": 3}[op]
    return {"bytes": vectors * 2 * mn * 8, "flops": 0.0}


# ------------------------------------------------------------------------------------------
# the same quantities in 64 bits, by dense transforms and direct solves in time
# ------------------------------------------------------------------------------------------
def _basis(case):
    """1D eigenvectors V (columns), V^-1 and eigenvalues of the second difference a K."""
    N, f8 = case["N"], dict(dtype=torch.float64, device="cuda")
    if case["bc"] == "neumann":
        L = N - 1
        k = torch.arange(N, **f8)
        V = torch.cos(PI * torch.remainder(torch.outer(k, k), 2 * L) / L)
        w = torch.ones(N, **f8)
        w[0] = w[-1] = 0.5
        inverse = (2.0 / L) * w[:, None] * V * w[None, :]
    else:
        L = N + 1
        k = torch.arange(1, N + 1, **f8)
        V = math.sqrt(2.0 / L) * torch.sin(PI * torch.remainder(torch.outer(k, k), 2 * L) / L)
        inverse = V
    kappa = case["a"] * 4.0 * L * L * torch.sin(PI * k / (2 * L)) ** 2
    return V, inverse, kappa


def _both(M, u):
    """M applied along both spatial axes of u (..., N, N)."""
    return torch.matmul(torch.matmul(M, u), M.T)


def _solve_exact(case, seed):
    """y and p from the optimality system itself, mode by mode: with u = sqrt(gamma) y and v = p,
        d u_t - e u_{t-1} - alpha (theta v_t + (1 - theta) v_{t+1}) = sqrt(gamma) f~_t
        alpha (theta u_t + (1 - theta) u_{t-1}) + d v_t - e v_{t+1}  = g~_t,
    d = 1 + theta tau kappa, e = 1 - (1 - theta) tau kappa: block tridiagonal in time (2 x 2 blocks)."""
    N, n, th, gamma = case["N"], case["n"], case["theta"], case["gamma"]
    tau = 1.0 / n
    alpha = tau / math.sqrt(gamma)
    V, inverse, kappa = _basis(case)
    g, f = (s.reshape(n + 1, N, N) for s in _samples(case, seed))
    r1 = _both(inverse, math.sqrt(gamma) * tau * (th * f[1:] + (1 - th) * f[:-1]))
    r2 = _both(inverse, tau * (th * g[:-1] + (1 - th) * g[1:]))
    c = tau * (kappa[:, None] + kappa[None, :])
    d, e, om = 1.0 + th * c, 1.0 - (1 - th) * c, 1.0 - th
    # forward elimination.  The blocks above the diagonal have one nonzero column (v_{t+1}), so each
    # step keeps two factors su, sv with u_t = r1_t - su v_{t+1}, v_t = r2_t - sv v_{t+1}.
    su, sv = torch.empty_like(r1), torch.empty_like(r1)
    a, b = d.clone(), torch.full_like(d, -alpha * th)       # current diagonal block [[a, b], [c0, d0]]
    c0, d0 = torch.full_like(d, alpha * th), d.clone()
    for t in range(n):
        if t:
            # u_{t-1} = r1 - su v_t enters through the lower block [[-e, 0], [alpha om, 0]]
            r1[t] += e * r1[t - 1]
            r2[t] -= alpha * om * r1[t - 1]
            b = -alpha * th + e * su[t - 1]
            d0 = d - alpha * om * su[t - 1]
        det = a * d0 - b * c0
        u1, u2 = -alpha * om, -e
        su[t] = (d0 * u1 - b * u2) / det
        sv[t] = (a * u2 - c0 * u1) / det
        q1, q2 = r1[t].clone(), r2[t].clone()
        r1[t] = (d0 * q1 - b * q2) / det
        r2[t] = (a * q2 - c0 * q1) / det
    for t in range(n - 2, -1, -1):
        r1[t] -= su[t] * r2[t + 1]
        r2[t] -= sv[t] * r2[t + 1]
    return {"y": (_both(V, r1) / math.sqrt(gamma)).reshape(-1), "p": _both(V, r2).reshape(-1)}


def _shift(u, by):
    """u one time level later (by = 1) or earlier (by = -1), zero beyond the ends."""
    out = torch.zeros_like(u)
    if by > 0:
        out[1:] = u[:-1]
    else:
        out[:-1] = u[1:]
    return out


def _product_exact(case, x, op):
    N, n, th = case["N"], case["n"], case["theta"]
    tau = 1.0 / n
    alpha = tau / math.sqrt(case["gamma"])
    x1, x2 = x.reshape(2, n, N, N)
    scale = case["a"] * tau * (N + 1) ** 2

    def stencil(u):
        pad = torch.nn.functional.pad(u, (1, 1, 1, 1))
        return scale * (4.0 * u - pad[:, 1:-1, :-2] - pad[:, 1:-1, 2:] - pad[:, :-2, 1:-1] - pad[:, 2:, 1:-1])

    z, w = x1.clone(), x2.clone()
    if th != 1.0:
        for t in range(n):
            z[t] = (x1[t] - ((1 - th) * z[t - 1] if t else 0.0)) / th
        for t in range(n - 1, -1, -1):
            w[t] = (x2[t] - ((1 - th) * w[t + 1] if t + 1 < n else 0.0)) / th
    row_t = z - _shift(z, 1) + stencil(x1) - alpha * x2
    row_tt = w - _shift(w, -1) + stencil(x2) + alpha * x1
    return torch.stack([row_tt, row_t] if op == "A" else [row_t, row_tt]).reshape(-1)


def _apply_exact(case, x):
    """P^-1 x by dense sine transforms and the complex FFT in time (real part)."""
    N, n, th = case["N"], case["n"], case["theta"]
    tau = 1.0 / n
    alpha = tau / math.sqrt(case["gamma"])
    V, inverse, kappa = _basis(case)
    t = torch.arange(n, dtype=torch.float64, device="cuda")
    twist = torch.polar(torch.ones_like(t), -case["zeta"] * t / n)[:, None, None]
    h = torch.fft.fft(_both(inverse, x.reshape(2, n, N, N)) * twist, dim=1)
    turn = torch.polar(torch.ones_like(t), -(case["zeta"] + 2.0 * PI * t) / n)
    lam = ((1.0 - turn) / (th + (1.0 - th) * turn))[:, None, None] + tau * (kappa[:, None] + kappa[None, :])
    size = lam.real ** 2 + lam.imag ** 2 + alpha * alpha
    if case["kind"] == "abs_ps":
        h = h / torch.sqrt(size)
    else:
        h = torch.stack([(lam.conj() * h[0] + alpha * h[1]) / size, (lam * h[1] - alpha * h[0]) / size])
    return _both(V, (torch.fft.ifft(h, dim=1) * twist.conj()).real).reshape(-1)


def exact(case, seed):
    op = case["op"]
    if op == "batch":
        return [_solve_exact(m, seed + 101 * k) for k, m in enumerate(_members(case))]
    if case["variable_a"]:
        return None              # no transform diagonalises it: the direct solve would take minutes
    if op == "solve":
        return _solve_exact(case, seed)
    if op == "host":
        # x carries sqrt(gamma) y and p (theta = 1: no change of variables)
        s = _solve_exact(case, seed)
        return {"x": torch.cat([math.sqrt(case["gamma"]) * s["y"], s["p"]])}
    x = _vector(2 * case["N"] ** 2 * case["n"], seed)
    if op == "apply":
        return {"y": _apply_exact(case, x)}
    if op == "product":
        return {"y": _product_exact(case, x, "A" if case["theta"] == 1.0 else "Ahat")}
    r = _vector(x.numel(), seed + 50021)
    out = _product_exact(case, x, "A") / BETA - (BETA / OLDB) * r
    return {"out": out, "dot": float(torch.dot(x, out)) / BETA}

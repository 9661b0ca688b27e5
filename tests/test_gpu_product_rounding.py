"""Rounding error of the theta < 1 product (csrc/matvec.cu, march_block) against extended precision: no
larger than when every term is formed on its own in FP64 with FMAs,
    z_t = (u_t - (1-theta) z_{t-1})/theta,   out = ((z_t - z_{t-1}) + tau K u_t) -/+ alpha (other half),
evaluated here.  Both relative 2-norm errors are averages over more than 10^5 roundings, which agree to
about 1/sqrt(10^5); 2% is allowed."""
import numpy as np
import pytest
import torch

import synth
from oracle import discretisation as ds

pytestmark = pytest.mark.gpu
L = np.longdouble


def fma(a, b, c):
    return (L(1) * a * b + c).astype(np.float64)


def products(prob, x, edges, neumann):
    """A_hat x with every term on its own in FP64, and in extended precision from the same coefficients."""
    N, n, th = prob.N, prob.n, prob.theta
    tau, h = 1.0 / n, 1.0 / (N - 1 if neumann else N + 1)
    alpha, c = tau / np.sqrt(prob.gamma), tau / (h * h)
    if edges is not None:
        e = c * edges
        ax, ay = e[:N * (N + 1)].reshape(N, N + 1), e[N * (N + 1):].reshape(N + 1, N)
        dg = ((ax[:, :-1] + ax[:, 1:]) + ay[:-1]) + ay[1:]

    def neighbours(u):
        p = np.pad(u, 1, mode="reflect" if neumann else "constant")
        return p[1:-1, :-2], p[1:-1, 2:], p[:-2, 1:-1], p[2:, 1:-1]

    def stencil64(u):
        l, r, d, t = neighbours(u)
        if edges is None:
            return fma(-c, (l + r) + (d + t), 4.0 * c * u)
        return fma(dg, u, -fma(ay[1:], t, fma(ay[:-1], d, fma(ax[:, 1:], r, ax[:, :-1] * l))))

    def stencil(u):
        l, r, d, t = neighbours(u)
        if edges is None:
            return L(c) * (4 * u - l - r - d - t)
        return dg * u - ax[:, :-1] * l - ax[:, 1:] * r - ay[:-1] * d - ay[1:] * t

    def march(u, w, sign, order):
        out64, out = np.empty_like(u), np.empty(u.shape, dtype=L)
        z64 = np.zeros_like(u[0])
        z = np.zeros(u[0].shape, dtype=L)
        for t in order:
            new64 = fma(-(1.0 - th), z64, u[t]) * (1.0 / th)
            out64[t] = fma(sign * alpha, w[t], (new64 - z64) + stencil64(u[t]))
            new = (u[t] - (1 - L(th)) * z) / L(th)
            out[t] = new - z + stencil(u[t].astype(L)) + sign * L(alpha) * w[t]
            z64, z = new64, new
        return out64, out

    x1, x2 = x.reshape(2, n, N, N)
    a, b = march(x1, x2, -1, range(n)), march(x2, x1, 1, range(n - 1, -1, -1))
    return np.concatenate([a[0].ravel(), b[0].ravel()]), np.concatenate([a[1].ravel(), b[1].ravel()])


@pytest.mark.parametrize("theta", [0.5, 0.7, 0.9])
@pytest.mark.parametrize("N,n,grid", [(63, 16, "dirichlet"), (255, 4, "dirichlet"), (65, 16, "neumann"), (63, 16, "variable"),
                                      (31, 128, "variable")])
def test_error_no_larger_than_with_separate_terms(N, n, grid, theta):
    from paper_2406_00952_gb300 import _build
    _build.build()
    import paper_2406_00952_gb300 as P
    edges = synth.variable_coefficient_edges(N) if grid == "variable" else None
    bc = "neumann" if grid == "neumann" else "dirichlet"
    prob = ds.Problem(N, n, theta, 1e-3, a_edges=edges, bc=bc)
    x = synth.random_vector(2 * N * N * n, seed=N + n)
    out = P.Problem(N, n, theta, 1e-3, a_edges=edges, bc=bc).matvec(torch.from_numpy(x).cuda(), op="Ahat").cpu().numpy()
    separate, exact = products(prob, x, edges, grid == "neumann")
    err = [float(np.linalg.norm((v - exact).astype(np.float64))) for v in (out, separate)]
    assert err[0] <= 1.02 * err[1], err

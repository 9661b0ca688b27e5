"""A profiled solve (profile=True times every preconditioner apply alone) gives the iterates of the same
solve without it, bit for bit: MINRES's residual update and inner product, which other solves run inside
the preconditioner's passes, have the same values in the same order beside them."""
import math

import numpy as np
import pytest
import torch

import synth
from oracle import discretisation as ds
from oracle import operators as op

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    from paper_2406_00952_gb300 import _build
    _build.build()
    import paper_2406_00952_gb300 as P
    return P


def dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


@pytest.mark.parametrize("precision,kind", [("mixed", "abs_ps"), ("mixed", "pms"), ("mixed", "none"), ("fp64", "abs_ps")])
@pytest.mark.parametrize("N,n", [(7, 8), (15, 2), (23, 16), (31, 16), (47, 8), (63, 4), (95, 8), (127, 4), (191, 2),
                                 (255, 4), (383, 2), (511, 2)])
def test_minres(P, N, n, precision, kind):
    prob = ds.Problem(N, n, 1.0, 1e-2)
    b = dev(ds.rhs_minres(prob, synth.random_target(N, n, seed=9), synth.manufactured_source(N, n))
            + 1e-3 * synth.random_vector(2 * prob.m * n, seed=10))
    gp = P.Problem(N, n, 1.0, 1e-2, precision=precision)
    plain, ip = gp.solve(b, precond=kind, method="minres", fixed_iterations=9)
    timed, it = gp.solve(b, precond=kind, method="minres", fixed_iterations=9, profile=True)
    assert it["precond_ms"] > 0.0 and ip["precond_ms"] == 0.0
    assert torch.equal(plain, timed)


@pytest.mark.parametrize("N,n", [(63, 32), (255, 16)])
def test_minres_residuals_below_the_fp32_range(P, N, n):
    """A residual with FP32 subnormal values, which the passes convert on a path of their own.  With a point
    source of a size at which P^{-1} b survives in FP32 only around it, the first residual is
    -(alfa/beta) b elsewhere: b there is chosen so that this lies below 2^-126."""
    prob = ds.Problem(N, n, 1.0, 1e-2)
    m, rng = prob.m, np.random.Generator(np.random.PCG64(3))
    b = np.zeros(2 * m * n)
    at = (n // 2) * m + (N // 2) * N + N // 2
    b[at] = 1.0
    gp = P.Problem(N, n, 1.0, 1e-2, precision="mixed")
    peak = float(gp.precond_apply(dev(b)).abs().max())
    back = np.ldexp(rng.uniform(-1.0, 1.0, b.size), -136)
    back[at] = 0.0
    b = np.ldexp(b + back, -146 - math.frexp(peak)[1])
    y = gp.precond_apply(dev(b)).cpu().numpy()
    beta = math.sqrt(b @ y)
    q = op.matvec_A(prob, y / beta)
    r1 = q - (y @ q) / beta / beta * b
    tiny = (np.abs(r1) < 2.0 ** -126) & (r1 != 0.0)
    assert beta > 0.0 and np.count_nonzero(tiny) > b.size // 8, (beta, np.count_nonzero(tiny))
    plain, _ = gp.solve(dev(b), fixed_iterations=3)
    timed, _ = gp.solve(dev(b), fixed_iterations=3, profile=True)
    assert np.all(np.isfinite(plain.cpu().numpy())) and torch.equal(plain, timed)

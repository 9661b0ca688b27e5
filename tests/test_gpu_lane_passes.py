"""The one-line-per-lane preconditioner passes (csrc/precond_lane.cuh) against the FP64 oracle: every
spatial line length with both boundary conditions (ragged last tiles, the smallest and the largest
grid), every time line with zeta = pi and another zeta, and the buffers their layouts depend on.

Tolerances are those of the parity tests: FP64 1e-12, FP32 2e-6, each on the relative 2-norm and the
relative max-norm error."""
import math

import numpy as np
import pytest
import torch

import synth
from closeness import assert_close
from oracle import discretisation as ds
from oracle import operators as op
from oracle import precond as pc

pytestmark = pytest.mark.gpu
ORACLE = {"abs_ps": pc.apply_abs_ps_inv, "ps": pc.apply_ps_inv, "pms": pc.apply_pms_inv}
TOL = {"fp64": 1e-12, "mixed": 2e-6}


@pytest.fixture(scope="module")
def P():
    from paper_2406_00952_gb300 import _build
    _build.build()
    import paper_2406_00952_gb300 as P
    return P


def dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def check(P, N, n, theta, zeta, bc, kind):
    a = 1e-3 if bc == "neumann" else 1.0
    prob = ds.Problem(N, n, theta, 1e-3, zeta=zeta, bc=bc, a0=a)
    v = synth.random_vector(2 * prob.m * n, seed=900 + N + n)
    ref = ORACLE[kind](prob, v)
    gp = P.Problem(N, n, theta, 1e-3, zeta=zeta, bc=bc, a=a)
    for precision, tol in TOL.items():
        assert_close(gp.precond_apply(dev(v), kind=kind, precision=precision).cpu().numpy(), ref, tol, what=precision)
        t = dev(v)                                                   # in place
        gp.precond_apply(t, out=t, kind=kind, precision=precision)
        assert_close(t.cpu().numpy(), ref, tol, what=precision + " in place")
    gp.close()


@pytest.mark.parametrize("L", [16, 24, 32, 48, 64, 96, 128, 192, 256, 384, 512])
@pytest.mark.parametrize("bc", ["dirichlet", "neumann"])
def test_spatial_lines(P, L, bc):
    neu = bc == "neumann"
    check(P, L + 1 if neu else L - 1, 4 if L < 256 else 2, 0.5, math.pi, bc, "ps" if neu else "pms")


@pytest.mark.parametrize("n", [2, 4, 8, 16, 32, 64, 128, 256, 512, 1024])
@pytest.mark.parametrize("zeta", [math.pi, 0.7], ids=["pi", "0.7"])
@pytest.mark.parametrize("kind", ["abs_ps", "ps", "pms"])
def test_time_lines(P, n, zeta, kind):
    check(P, 23, n, 1.0, zeta, "dirichlet", kind)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("N,n", [(47, 32), (255, 4), (511, 2)])
def test_output_aligned_to_eight_bytes_only(P, precision, N, n):
    """The FP64 passes park an intermediate result in the output vector, FP32 ones write it in FP64."""
    prob = ds.Problem(N, n, 1.0, 1e-2)
    v = synth.random_vector(2 * prob.m * n, seed=77 + N)
    buf = torch.zeros(v.size + 1, dtype=torch.float64, device="cuda")
    out = P.Problem(N, n, 1.0, 1e-2).precond_apply(dev(v), out=buf[1:], kind="abs_ps", precision=precision)
    assert out.data_ptr() % 16 == 8 and float(buf[0]) == 0.0
    assert_close(out.cpu().numpy(), pc.apply_abs_ps_inv(prob, v), TOL[precision])


def test_values_outside_the_fp32_range(P):
    """Infinities and NaN reach the output, values past the FP32 range overflow as the conversion
    instruction does, and a line of FP32 subnormals keeps them."""
    N, n = 47, 16
    gp = P.Problem(N, n, 1.0, 1e-2, precision="mixed")
    for bad in (float("inf"), float("nan"), 1e300):
        v = synth.random_vector(2 * N * N * n, seed=5)
        v[1234] = bad
        assert not np.all(np.isfinite(gp.precond_apply(dev(v), kind="abs_ps").cpu().numpy()))
    v = synth.random_vector(2 * N * N * n, seed=6)
    one = gp.precond_apply(dev(v), kind="abs_ps").cpu().numpy()
    tiny = gp.precond_apply(dev(v * 2.0 ** -120), kind="abs_ps").cpu().numpy() * 2.0 ** 120
    # intermediate values near 2^-120 times the weights stay above the FP32 subnormal spacing 2^-149:
    # 2^-29 relative to the input, times the growth of at most 4 lines' rounding
    assert np.linalg.norm(tiny - one) <= 2.0 ** -20 * np.linalg.norm(v)


def test_batch_of_different_zetas(P):
    """Instances of one line length and different omega share launches; each keeps its own twist."""
    zetas, N, n = (0.3, math.pi / 2, 2.1), 31, 64
    probs, bs, gps = [], [], []
    for k, z in enumerate(zetas):
        prob = ds.Problem(N, n, 1.0, 1e-3, zeta=z)
        probs.append(prob)
        bs.append(ds.rhs_minres(prob, synth.random_target(N, n, seed=80 + k), synth.manufactured_source(N, n)))
        gps.append(P.Problem(N, n, 1.0, 1e-3, zeta=z, precision="mixed"))
    xs, infos = P.batch_solve(gps, [dev(b) for b in bs], tol=1e-8)
    for prob, b, gp, x, info in zip(probs, bs, gps, xs, infos):
        assert np.linalg.norm(b - op.matvec_A(prob, x.cpu().numpy())) <= 1.5e-8 * np.linalg.norm(b)
        _, alone = P.batch_solve([gp], [dev(b)], tol=1e-8)
        assert alone[0]["iterations"] == info["iterations"]


@pytest.mark.parametrize("N,n", [(15, 2), (31, 16), (47, 8), (95, 4), (127, 4), (191, 2), (255, 4), (383, 2), (511, 2)])
def test_residual_update_and_inner_product_in_the_passes(P, N, n):
    """A mixed solve forms MINRES's residual in pass 1 and its inner product in pass 5; a profiled one
    keeps both in kernels of their own.  The same residual bit for bit, the sum in another order: iterates
    after 5 steps agree to the rounding of beta carried through the recurrences (1e-12), for sizes with
    every line length and ragged tiles."""
    prob = ds.Problem(N, n, 1.0, 1e-2)
    b = dev(ds.rhs_minres(prob, synth.random_target(N, n, seed=9), synth.manufactured_source(N, n))
            + 1e-3 * synth.random_vector(2 * prob.m * n, seed=10))
    gp = P.Problem(N, n, 1.0, 1e-2, precision="mixed")
    fused, i1 = gp.solve(b, fixed_iterations=5)
    apart, i2 = gp.solve(b, fixed_iterations=5, profile=True)
    assert i1["launches"] < i2["launches"]
    assert_close(fused.cpu().numpy(), apart.cpu().numpy(), 1e-12)

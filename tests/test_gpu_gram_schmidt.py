"""Gram-Schmidt of FGMRES (csrc/krylov.cu): every basis count up to the restart limit through iterates
that have not converged (no preconditioner), against the oracle's FGMRES; a solution vector
aligned to eight bytes only.  Iterates of one algorithm in FP64: 1e-10."""
import numpy as np
import pytest
import torch

import synth
from closeness import assert_close
from oracle import discretisation as ds
from oracle import krylov as kr
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


@pytest.mark.parametrize("k", [1, 2, 7, 8, 9, 16, 17, 25, 31, 32])
@pytest.mark.parametrize("N,n", [(15, 16), (47, 8)])
def test_unpreconditioned_iterates(P, N, n, k):
    prob = ds.Problem(N, n, 0.5, 1e-2)
    b = ds.rhs_gmres(prob, synth.random_target(N, n, seed=3), synth.manufactured_source(N, n))
    b = b + 1e-3 * np.linalg.norm(b) / np.sqrt(b.size) * synth.random_vector(b.size, seed=4)
    xo, _ = kr.fgmres(lambda z: op.matvec_A_hat(prob, z), b, lambda r: r, restart=32, fixed_iterations=k)
    gp = P.Problem(N, n, 0.5, 1e-2)
    buf = torch.zeros(b.size + 1, dtype=torch.float64, device="cuda")
    x, info = gp.solve(dev(b), x=buf[1:], method="gmres", precond="none", restart=32, fixed_iterations=k)
    assert info["iterations"] == k and x.data_ptr() % 16 == 8
    assert_close(x.cpu().numpy(), xo, 1e-10, what=k)
    gp.close()


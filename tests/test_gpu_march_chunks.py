"""The theta < 1 product in parts of the time range (csrc/matvec.cu, march_block) against the FP64
oracle: grids that take 8, 4, 2 and 1 parts (by their column count), the fewest steps a part may have,
ragged last blocks, both operators, Neumann grids, a variable coefficient, and theta other than 1/2.
Tolerance 1e-13, as for every FP64 product."""
import numpy as np
import pytest
import torch

import synth
from closeness import assert_close
from oracle import discretisation as ds
from oracle import operators as op

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,n", [(1, 2), (2, 8), (7, 32), (63, 64), (95, 32), (127, 16), (191, 8), (255, 4)])
@pytest.mark.parametrize("theta", [0.5, 0.7])
@pytest.mark.parametrize("grid", ["dirichlet", "neumann", "variable"])
def test_product(N, n, theta, grid):
    from paper_2406_00952_gb300 import _build
    _build.build()
    import paper_2406_00952_gb300 as P
    if grid == "neumann":
        N = max(N, 2) + (2 if N % 2 else 3)          # N - 1 = 2^a 3^b
        if N - 1 not in (4, 8, 64, 96, 128, 192, 256):
            pytest.skip("no Neumann grid of this size")
    edges = synth.variable_coefficient_edges(N) if grid == "variable" else None
    if grid == "variable" and (N + 1) & N:
        pytest.skip("a variable coefficient needs N = 2^k - 1")
    bc = "neumann" if grid == "neumann" else "dirichlet"
    prob = ds.Problem(N, n, theta, 1e-3, a_edges=edges, bc=bc)
    v = synth.random_vector(2 * prob.m * n, seed=40 + N + n)
    gp = P.Problem(N, n, theta, 1e-3, a_edges=edges, bc=bc)
    for name, f in (("A", op.matvec_A), ("Ahat", op.matvec_A_hat)):
        out = gp.matvec(torch.from_numpy(v).cuda(), op=name).cpu().numpy()
        assert_close(out, f(prob, v), 1e-13, what=name)
    gp.close()

"""A mixed-precision result does not depend on which problems share its launches, bit for bit: MINRES
instances whose grids have the one-line-per-lane passes (where the residual update and the inner product
run inside the preconditioner) beside grids that have none (N + 1 < 16), in a batch and in the server."""
import numpy as np
import pytest
import torch

import synth
from oracle import discretisation as ds

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    from paper_2406_00952_gb300 import _build
    _build.build()
    import paper_2406_00952_gb300 as P
    return P


def rhs(N, n, gamma, seed):
    return ds.rhs_minres(ds.Problem(N, n, 1.0, gamma), synth.random_target(N, n, seed=seed), synth.manufactured_source(N, n))


@pytest.mark.parametrize("graphs", [True, False])
@pytest.mark.parametrize("shapes", [((63, 16, 1e-2), (7, 64, 1e-3)),
                                    ((5, 8, 1e-2), (47, 32, 1e-4), (23, 8, 1e-1), (11, 128, 1e-5), (191, 4, 1e-3))])
def test_batch(P, shapes, graphs):
    gps = [P.Problem(N, n, 1.0, gamma, precision="mixed") for N, n, gamma in shapes]
    bs = [torch.from_numpy(rhs(N, n, gamma, 20 + k)).cuda() for k, (N, n, gamma) in enumerate(shapes)]
    xs, infos = P.batch_solve(gps, bs, tol=1e-10, graphs=graphs)
    for gp, b, x, info in zip(gps, bs, xs, infos):
        alone, ia = P.batch_solve([gp], [b], tol=1e-10, graphs=graphs)
        assert ia[0]["iterations"] == info["iterations"] and ia[0]["refinements"] == info["refinements"]
        assert torch.equal(alone[0], x), (gp.N, gp.n)


def test_server_requests_without_the_passes_come_and_go(P):
    """Small requests with a zero right-hand side are admitted during a large one's solve, each present
    in its launches for a step."""
    from paper_2406_00952_gb300 import serve

    def run(guests):
        srv = serve.Server(1 << 30, max_slots=2, tol=1e-12)
        b = torch.from_numpy(rhs(95, 32, 1e-3, 5) + 1e-4 * synth.random_vector(2 * 95 * 95 * 32, seed=7)).pin_memory()
        x = torch.full_like(b, float("nan")).pin_memory()
        zero = torch.zeros(2 * 7 * 7 * 8, dtype=torch.float64).pin_memory()
        srv.submit(95, 32, 1.0, 1e-3, b, x, 0)
        done = {}
        for step in range(400):
            if guests and step >= 2:
                srv.submit(7, 8, 1.0, 1e-1, zero, torch.empty_like(zero).pin_memory(), step)
            done.update({c.tag: c for c in srv.step()[0]})
            if 0 in done:
                break
        srv.close()
        assert done[0].status == 0 and len(done) >= (3 if guests else 1), done
        return x.numpy().copy(), done[0].iterations

    x0, its0 = run(False)
    x1, its1 = run(True)
    assert its0 == its1 and np.array_equal(x0, x1)

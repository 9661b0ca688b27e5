"""Batches whose instances take different FP32 preconditioner kernels: one line per lane (the default),
pipelined with and without the n = 512 hand-off, pipelined time with tile spatial passes, tile kernels,
and a grid that has tile kernels only (N + 1 = 8), in one MINRES and one GMRES group.  The kernels are
pinned with tune_select.  Each result is that of the instance alone, bit for bit, and meets the tolerance in
the oracle's FP64 residual."""
import numpy as np
import pytest
import torch

import synth
from oracle import discretisation as ds
from oracle import operators as op

pytestmark = pytest.mark.gpu
LAST = -1          # the pipelined kernels in their default shapes end the list

# N, n, theta, gamma, configuration (0: the default)
MIXES = {
    "minres": [(31, 512, 1.0, 1e-2, LAST), (31, 512, 1.0, 1e-4, 1), (31, 128, 1.0, 1e-3, LAST), (63, 64, 1.0, 1e-4, LAST),
               (15, 64, 1.0, 1e-2, LAST), (47, 32, 1.0, 1e-3, 2), (63, 64, 1.0, 1e-2, 0), (95, 16, 1.0, 1e-1, 0),
               (7, 64, 1.0, 1e-2, 0)],
    "gmres": [(31, 128, 0.5, 1e-3, LAST), (47, 32, 0.5, 1e-3, 2), (63, 64, 0.5, 1e-2, 0), (15, 64, 0.5, 1e-4, 1),
              (7, 32, 0.5, 1e-2, 0)],
    "both": [(63, 64, 1.0, 1e-2, LAST), (63, 64, 1.0, 1e-2, 0), (31, 32, 0.5, 1e-3, 0), (31, 32, 0.5, 1e-3, LAST),
             (7, 16, 1.0, 1e-3, 0), (11, 16, 0.5, 1e-3, 0)],
}


@pytest.mark.parametrize("graphs", [True, False])
@pytest.mark.parametrize("mix", MIXES)
def test_batch(mix, graphs):
    from paper_2406_00952_gb300 import _build
    _build.build()
    import paper_2406_00952_gb300 as P
    insts, kinds = [], set()
    for k, (N, n, theta, gamma, pin) in enumerate(MIXES[mix]):
        prob = ds.Problem(N, n, theta, gamma)
        g, f = synth.random_target(N, n, seed=40 + k), synth.manufactured_source(N, n)
        b = ds.rhs_minres(prob, g, f) if theta == 1.0 else ds.rhs_gmres(prob, g, f)
        gp = P.Problem(N, n, theta, gamma, precision="mixed")
        if pin:
            info = gp.tune_select(gp.tune_select(-1)["candidates"] - 1 if pin == LAST else pin)
            kinds.add((info["pipelined_dst"], info["pipelined_time"], info["time_major_handoff"]))
        insts.append((prob, b, gp))
    if mix == "minres":
        assert kinds >= {(1, 1, 1), (1, 1, 0), (0, 1, 0), (0, 0, 0)}, kinds
    bs = [torch.from_numpy(b).cuda() for _, b, _ in insts]
    xs, infos = P.batch_solve([gp for _, _, gp in insts], bs, tol=1e-8, restart=16, graphs=graphs)
    for (prob, b, gp), bd, x, info in zip(insts, bs, xs, infos):
        A = op.matvec_A if prob.theta == 1.0 else op.matvec_A_hat
        assert np.linalg.norm(b - A(prob, x.cpu().numpy())) <= 1.5e-8 * np.linalg.norm(b)
        alone, ia = P.batch_solve([gp], [bd], tol=1e-8, restart=16, graphs=graphs)
        assert ia[0]["iterations"] == info["iterations"]
        assert torch.equal(alone[0], x), (prob.N, prob.n, prob.theta)

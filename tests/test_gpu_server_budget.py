"""The workspace of an FP64 request in the server: eleven vectors, the preconditioner's scratch of one
more, and the tables; the padded scratch of the FP32 passes is not part of it."""
import pytest
import torch

import synth
from oracle import discretisation as ds

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,n", [(15, 16), (47, 64)])
def test_fp64_request_in_twelve_vectors(N, n):
    from paper_2406_00952_gb300 import _build
    _build.build()
    from paper_2406_00952_gb300 import serve
    b = torch.from_numpy(ds.rhs_minres(ds.Problem(N, n, 1.0, 1e-2), synth.random_target(N, n, seed=1),
                                       synth.manufactured_source(N, n))).pin_memory()
    srv = serve.Server(12 * b.numel() * 8 + (64 << 10), max_slots=1, precision="fp64")
    x = torch.empty_like(b).pin_memory()
    srv.submit(N, n, 1.0, 1e-2, b, x, 0)
    done = []
    for _ in range(200):
        done += srv.step()[0]
        if done:
            break
    srv.close()
    assert done and done[0].status == 0 and done[0].relres <= 1e-8

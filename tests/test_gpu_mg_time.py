"""The multigrid route's fused kernels (csrc/mg.cu).  The time transforms at the line lengths and column
counts where their tiles end raggedly: against the FP64 oracle, and with values at the edge of the FP32
range, which take the conversions' rare branch.  Tolerances as for the route's other parity tests: 1e-12 in
FP64, 5e-6 in FP32.  For the tiny values add the spacing of FP32 subnormals, 2^-149, in the input and the
result: 2e-7 of results of size 1e-38."""
import pytest
import torch

import synth
from closeness import assert_close
from oracle import discretisation as ds
from oracle import precond as pc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1.0, 1e-36])
@pytest.mark.parametrize("N,n", [(3, 4), (7, 32), (3, 128), (7, 256), (3, 512)])
@pytest.mark.parametrize("kind", ["ps", "pms"])
def test_transforms(kind, N, n, scale):
    import paper_2406_00952_gb300 as P
    a = synth.variable_coefficient_edges(N)
    prob = ds.Problem(N, n, 1.0, 1e-3, a_edges=a)
    v = synth.random_vector(2 * prob.m * n, seed=70 + N + n)
    ref = pc.apply_mg_ps_inv(prob, v, cycles=2) if kind == "ps" else pc.apply_pms_inv(prob, v, cycles=2)
    gp = P.Problem(N, n, 1.0, 1e-3, a_edges=a, mg_cycles=2)
    x = torch.from_numpy(v * scale).cuda()
    out64 = gp.precond_apply(x, kind=kind, precision="fp64").cpu().numpy() / scale
    out32 = gp.precond_apply(x, kind=kind, precision="mixed").cpu().numpy() / scale
    gp.close()
    assert_close(out64, ref, 1e-12, what="fp64")
    assert_close(out32, ref, 5e-6 if scale == 1.0 else 5.2e-6, what="fp32")


@pytest.mark.parametrize("cycles", [1, 3])
@pytest.mark.parametrize("N,n", [(1, 2), (7, 4), (31, 4), (63, 2), (127, 2)])
def test_smoothing(N, n, cycles):
    """The smoothing kernels on grids inside one tile, ending one point short of a tile, and of several tiles;
    one cycle (the result written) and three (added to the iterate)."""
    import paper_2406_00952_gb300 as P
    a = synth.variable_coefficient_edges(N)
    prob = ds.Problem(N, n, 0.5, 1e-3, a_edges=a)
    v = synth.random_vector(2 * prob.m * n, seed=90 + N + n)
    ref = pc.apply_mg_ps_inv(prob, v, cycles=cycles)
    gp = P.Problem(N, n, 0.5, 1e-3, a_edges=a, mg_cycles=cycles)
    out64 = gp.precond_apply(torch.from_numpy(v).cuda(), kind="ps", precision="fp64").cpu().numpy()
    out32 = gp.precond_apply(torch.from_numpy(v).cuda(), kind="ps", precision="mixed").cpu().numpy()
    gp.close()
    assert_close(out64, ref, 1e-12, what="fp64")
    assert_close(out32, ref, 5e-6, what="fp32")

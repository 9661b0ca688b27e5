"""The configurations behind the indices of pcb_tune_select: a caller that pinned one of the pipelined
or tile kernels by its index keeps getting it; index 0 is the default, and the pipelined kernels' own
default shapes are the last of the list."""
import pytest

pytestmark = pytest.mark.gpu
FIELDS = ("pipelined_dst", "pipelined_time", "time_major_handoff", "time512_blocks", "dst_lanes", "time_lanes", "tile_scale")

# (N, n, precision, bc): configurations 1, 2, ... in the order of FIELDS, then the last one.  The shapes'
# list before the one-line-per-lane passes, whose entry 0 is now the last.
SMALL = ([(0, 1, 0, 2, 32, 32, 1.0), (0, 0, 0, 2, 32, 32, 1.0), (0, 0, 0, 2, 32, 16, 1.0), (0, 1, 0, 2, 16, 32, 1.0),
          (0, 0, 0, 2, 16, 32, 1.0), (0, 0, 0, 2, 16, 16, 1.0), (0, 1, 0, 2, 32, 32, 0.5)], (1, 1, 0, 2, 32, 32, 1.0))
LISTS = {
    (255, 512, "mixed", "dirichlet"): ([(1, 1, 0, 2, 32, 32, 1.0), (1, 1, 1, 3, 32, 32, 1.0), (1, 1, 0, 3, 32, 32, 1.0),
                                        (1, 1, 1, 4, 32, 32, 1.0), (1, 1, 0, 4, 32, 32, 1.0), (0, 1, 0, 2, 32, 32, 1.0),
                                        (0, 0, 0, 2, 32, 32, 1.0)], (1, 1, 1, 2, 32, 32, 1.0)),
    (63, 64, "mixed", "dirichlet"): SMALL,
    (129, 128, "mixed", "neumann"): SMALL,
}


@pytest.mark.parametrize("key", LISTS)
def test_order(key):
    from paper_2406_00952_gb300 import _build
    _build.build()
    import paper_2406_00952_gb300 as P
    N, n, precision, bc = key
    gp = P.Problem(N, n, 0.5, 1e-2, precision=precision, bc=bc)
    count = gp.tune_select(-1)["candidates"]
    got = [tuple(gp.tune_select(k)[f] for f in FIELDS) for k in range(count)]
    first, last = LISTS[key]
    assert got[1:1 + len(first)] == first and got[-1] == last

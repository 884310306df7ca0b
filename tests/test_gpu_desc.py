"""GPU parity: the fast solve's descent levels on tiles (transforms of 2^13 and
more) at ragged nodes: a last node whose right child is empty (copied), holds
one root or is full, at levels with and without column passes, against the
quadratic solve."""
import random

import numpy as np
import pytest

from tests.gpuutil import d64, h64, rand_nodes, rand_res, zeros64
from tests.pyref import P63

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__ as ge
    from paper_2505_24256_gb300 import zr

    ge.build()
    c = zr.Context(P63)
    yield c
    c.close()


@pytest.mark.parametrize("T,S,offset", [(16385, 40, 0), (20000, 21, 1), (32768, 33, 0), (33000, 21, 1), (45057, 31, 0),
                                        (65537, 2, 1), (131071, 9, 0), (131073, 1, 0), (300001, 1, 1)])
def test_tile_levels_match_the_quadratic_solve(ctx, T, S, offset):
    rnd = random.Random(T + S)
    v, b = rand_nodes(rnd, T, P63), rand_res(rnd, (S, T), P63)
    b[0, :4] = [0, P63 - 1, 1, P63 - 2]
    dv, db = d64(v), d64(b)
    out = []
    for method in (ctx.SOLVE_FAST, ctx.SOLVE_QUADRATIC):
        c = zeros64(S, T)
        ctx.solve_method(method)
        try:
            ctx.vandermonde_solve([dict(T=T, S=S, offset=offset, v=dv, b=db, ldb=T, c=c, ldc=T)])
        finally:
            ctx.solve_method(0)
        out.append(h64(c))
    assert np.array_equal(out[0], out[1])

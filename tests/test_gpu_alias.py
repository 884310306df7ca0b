"""GPU parity: systems whose solution is written over their own nodes (the ABI
only forbids it over the right-hand sides), by each of the solves."""
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


# one CTA, several CTAs of a cluster, the O(T^2) kernels
@pytest.mark.parametrize("T", [20, 33, 200, 256, 300])
@pytest.mark.parametrize("S,row,offset", [(1, 0, 0), (1, 0, 1), (3, 2, 1)])
def test_solution_over_the_nodes(ctx, orc, T, S, row, offset):
    rnd = random.Random(T + S + offset)
    v, b = rand_nodes(rnd, T, P63), rand_res(rnd, (S, T), P63)
    want = orc.tvandermonde_solve(v, b, offset=offset)
    c, db = zeros64(S, T), d64(b)
    for _ in range(5):
        c[row] = d64(v)
        ctx.vandermonde_solve([dict(T=T, S=S, offset=offset, v=c[row], b=db, ldb=T, c=c, ldc=T)])
        assert np.array_equal(h64(c), want)

"""GPU parity: the fast solve's leaves on the tensor cores at the edges of
their tiles (128 roots), blocks (128 and 256 roots), k-steps (16), chunks (128)
and column groups (16 rows), against the oracle."""
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
    c.solve_method(c.SOLVE_FAST)
    yield c
    c.close()


@pytest.mark.parametrize("T,S,offset", [(1, 1, 0), (16, 15, 1), (17, 16, 0), (127, 3, 0), (129, 31, 1), (255, 17, 0),
                                        (2047, 15, 0), (2048, 16, 1), (2049, 2, 0), (2176, 32, 0), (2177, 33, 1),
                                        (2303, 63, 0), (2319, 1, 0)])
def test_leaf_edges(ctx, orc, T, S, offset):
    rnd = random.Random(100 * T + S)
    v, b = rand_nodes(rnd, T, P63), rand_res(rnd, (S, T), P63)
    if T > 4:
        v[0], v[1], b[0, :4] = P63 - 1, 1, [0, P63 - 1, 1, P63 - 2]
        if len(set(v.tolist())) < T:
            pytest.skip("nodes collide")
    c = zeros64(S, T)
    ctx.vandermonde_solve([dict(T=T, S=S, offset=offset, v=d64(v), b=d64(b), ldb=T, c=c, ldc=T)])
    assert np.array_equal(h64(c), orc.tvandermonde_solve(v, b, offset=offset))

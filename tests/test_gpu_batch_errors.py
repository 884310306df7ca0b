"""GPU: a call that cannot enqueue one of its entries leaves nothing under way on
other streams that the next call's tables and workspace could be laid over."""
import random

import numpy as np
import pytest

from tests.gpuutil import d64, h64, rand_nodes, rand_res, zeros64
from tests.pyref import P63

pytestmark = pytest.mark.gpu


def system(rnd, T, S):
    v, b = rand_nodes(rnd, T, P63), rand_res(rnd, (S, T), P63)
    return dict(T=T, S=S, offset=0, v=d64(v), b=d64(b), ldb=T, c=zeros64(S, T), ldc=T), v, b


def test_refused_entry_beside_small_and_fast_ones(orc):
    import __graft_entry__ as ge
    from paper_2505_24256_gb300 import zr

    ge.build()
    rnd = random.Random(3)
    # 128 right-hand sides of 300 unknowns have no kernel of the O(T^2) method
    refused = [system(rnd, *s)[0] for s in [(256, 32), (300, 128), (1, 2), (200, 20), (3000, 20)]]
    good = [system(rnd, *s) for s in [(40, 7), (700, 3), (256, 9), (2500, 20)]]
    want = [orc.tvandermonde_solve(v, b) for _, v, b in good]
    ctx = zr.Context(P63)
    for _ in range(8):
        with pytest.raises(zr.ZrError) as e:
            ctx.vandermonde_solve(refused)
        assert e.value.status == zr.INVALID_ARG
        ctx.vandermonde_solve([g[0] for g in good])
        for (d, _, _), w in zip(good, want):
            assert np.array_equal(h64(d["c"]), w)
            d["c"].zero_()
    ctx.close()

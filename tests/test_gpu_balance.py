"""GPU parity: the per-probe rational reconstruction of the balanced step at
the edges of its warp layout (16 and 32 coefficients, 32 and 64 samples) and
its failures, against the oracle."""
import random

import numpy as np
import pytest

from tests.gpuutil import d8, d64, h64, zeros8, zeros64
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


def horner(c, x):
    r = 0
    for a in reversed(c):
        r = (r * x + a) % P63
    return r


def problem(rnd, T, num, den, Sf):
    """Skeletons of T monomials x_0^i and, per probe, the values of a random
    fraction with numerator degree num and denominator degree den."""
    sk = np.zeros((T, 2), dtype=np.uint8)
    sk[:, 0] = np.arange(T)
    cs = rnd.sample(range(1, P63), Sf)
    f = np.zeros((Sf, T), dtype=np.uint64)
    for i in range(T):
        n = [rnd.randrange(1, P63) for _ in range(num + 1)]
        d = [rnd.randrange(1, P63) for _ in range(den + 1)]
        for s, c in enumerate(cs):
            f[s, i] = horner(n, c) * pow(horner(d, c), P63 - 2, P63) % P63
    return sk, cs, f, [rnd.randrange(1, P63)], np.array([rnd.randrange(1, P63) for _ in range(T)], dtype=np.uint64)


def run(ctx, sk, y, dN, dD, cs, f, dcoef):
    T = sk.shape[0]
    e, c = d8(sk), d64(dcoef)
    oN, oD = (zeros8(T * (dN + 1), 2), zeros64(T * (dN + 1))), (zeros8(T * (dD + 1), 2), zeros64(T * (dD + 1)))
    nN, nD = ctx.zippel_step_balanced(ctx.poly(2, T, e), ctx.poly(2, T, e, c), 1, d64(y), dN, dD, d64(cs), d64(f), T, 0,
                                      *oN, T * (dN + 1), *oD, T * (dD + 1))
    return [(a[:n].cpu().numpy(), h64(b[:n])) for (a, b), n in ((oN, nN), (oD, nD))]


@pytest.mark.parametrize("num,den,dN,dD", [(0, 0, 0, 0), (1, 0, 1, 0), (7, 8, 7, 8), (3, 15, 15, 15), (15, 15, 15, 15),
                                           (16, 2, 16, 2), (16, 16, 16, 16), (31, 31, 31, 31), (30, 31, 31, 31)])
@pytest.mark.parametrize("T", [1, 9])
def test_balanced_edges(ctx, orc, num, den, dN, dD, T):
    rnd = random.Random(1000 * num + 10 * den + T)
    Sf = 2 * max(dN, dD) + 2
    sk, cs, f, y, dcoef = problem(rnd, T, num, den, Sf)
    dprev = orc.zippel_probes(sk, dcoef, 1, y, [1], [1, 1], T)[0]
    bN, bD = orc.balance_probes(cs, f, dprev, dN, dD, T, T)
    want = [orc.zippel_step(sk, 1, y, cs[: b.shape[0]], b) for b in (bN, bD)]
    for (ge, gc), (we, wc) in zip(run(ctx, sk, y, dN, dD, cs, f, dcoef), want):
        assert np.array_equal(ge, we) and np.array_equal(gc, wc)


@pytest.mark.parametrize("deg", [3, 20])
def test_balanced_failures(ctx, deg):
    from paper_2505_24256_gb300 import zr

    rnd = random.Random(deg)
    Sf = 2 * deg + 2
    sk, cs, f, y, dcoef = problem(rnd, 9, deg, deg, Sf)

    def status(f, dN, dD):
        with pytest.raises(zr.ZrError) as e:
            run(ctx, sk, y, dN, dD, cs, f, dcoef)
        return e.value.status

    assert status(f, deg - 1, deg) == zr.DEGREE          # a numerator above its bound
    bad = f.copy()
    bad[:, 4] = [rnd.randrange(1, P63) for _ in range(Sf)]
    assert status(bad, deg, deg) == zr.DEGREE            # never closes within the samples
    bad[Sf - 1, 4] = bad[0, 4]
    assert status(bad, deg, deg) == zr.UNLUCKY           # one equal pair: a degenerate table
    run(ctx, sk, y, deg, deg, cs, f, dcoef)              # the context goes on

"""GPU parity over the whole range of primes a context takes (2^32 < p <
2^63): the solves, the evaluators, small entries, the balanced step and full
reconstructions, each against the oracle or the function it was made from."""
import random

import numpy as np
import pytest

from paper_2505_24256_gb300 import workloads as W
from tests.gpuutil import d8, d64, h64, rand_nodes, rand_res, zeros8, zeros64
from tests.pyref import P63

pytestmark = pytest.mark.gpu

# the smallest prime above 2^32, the largest below 2^40 and 2^46, the smallest
# above 2^46, and 2^63 - 25
PRIMES = [4294967311, 1099511627689, 70368744177643, 70368744177679, P63]


@pytest.fixture(scope="module", params=PRIMES)
def ctx(request):
    import __graft_entry__ as ge
    from paper_2505_24256_gb300 import zr

    ge.build()
    c = zr.Context(request.param)
    yield c
    c.close()


# one leaf block and several of them, leaves of 128 and of 256 roots
@pytest.mark.parametrize("T,S", [(100, 3), (300, 2), (2047, 1), (2177, 17)])
@pytest.mark.parametrize("offset", [0, 1])
def test_fast_solve(ctx, orc, T, S, offset):
    rnd = random.Random(T + S)
    v, b = rand_nodes(rnd, T, ctx.p), rand_res(rnd, (S, T), ctx.p)
    c = zeros64(S, T)
    ctx.solve_method(ctx.SOLVE_FAST)
    try:
        ctx.vandermonde_solve([dict(T=T, S=S, offset=offset, v=d64(v), b=d64(b), ldb=T, c=c, ldc=T)])
    finally:
        ctx.solve_method(0)
    assert np.array_equal(h64(c), orc.tvandermonde_solve(v, b, offset=offset, p=ctx.p))


# the O(T^2) solve, and an entry of one launch
@pytest.mark.parametrize("T,S", [(300, 5), (256, 32), (70, 3)])
def test_quadratic_solve(ctx, orc, T, S):
    rnd = random.Random(T + S)
    v, b = rand_nodes(rnd, T, ctx.p), rand_res(rnd, (S, T), ctx.p)
    c = zeros64(S, T)
    ctx.vandermonde_solve([dict(T=T, S=S, offset=1, v=d64(v), b=d64(b), ldb=T, c=c, ldc=T)])
    assert np.array_equal(h64(c), orc.tvandermonde_solve(v, b, offset=1, p=ctx.p))


# the integer kernel, the tensor cores (S T Tf = 5e7 and T (S + 4) Tf = 6e7),
# the transposed tree
@pytest.mark.parametrize("Tf,S,T,method", [(300, 5, 200, 0), (2000, 21, 1200, 0), (900, 5, 700, 2)])
@pytest.mark.parametrize("offset", [0, 1])
def test_probes(ctx, orc, Tf, S, T, method, offset):
    rnd = random.Random(Tf + S)
    nv, k = 5, 4
    exps = W.distinct_monomials_box(W.Stream(Tf, 1), Tf, nv, 9)
    coef, y, cs, z = (rand_res(rnd, (n,), ctx.p) for n in (Tf, k, S, nv))
    out = zeros64(S, T)
    ke, kc, ky, kcs, kz = d8(exps), d64(coef), d64(y), d64(cs), d64(z)
    ctx.solve_method(method)
    try:
        ctx.zippel_probes(ctx.poly(nv, Tf, ke, kc), k, ky, S, kcs, kz, T, offset, out, T)
    finally:
        ctx.solve_method(0)
    assert np.array_equal(h64(out), orc.zippel_probes(exps, coef, k, y, cs, z, T, offset, p=ctx.p))


@pytest.mark.parametrize("T,S", [(40, 6), (256, 21), (600, 4), (2100, 9)])
def test_step(ctx, orc, T, S):
    rnd = random.Random(T + S)
    nv, k = 5, 4
    skel = np.zeros((T, nv), dtype=np.uint8)
    skel[:, :k] = W.distinct_monomials_box(W.Stream(T, 1), T, k, 12)
    y, b = rand_res(rnd, (k,), ctx.p), rand_res(rnd, (S, T), ctx.p)
    cs = np.array(rnd.sample(range(1, ctx.p), S), dtype=np.uint64)
    oe, oc = zeros8(T * S, nv), zeros64(T * S)
    ks, ky, kcs, kb = d8(skel), d64(y), d64(cs), d64(b)
    n = ctx.zippel_step(ctx.poly(nv, T, ks), k, ky, S, kcs, kb, T, 0, oe, oc, T * S)
    we, wc = orc.zippel_step(skel, k, y, cs, b, p=ctx.p)
    assert n == we.shape[0]
    assert np.array_equal(oe[:n].cpu().numpy(), we) and np.array_equal(h64(oc[:n]), wc)


def needs_draws(ctx):
    if ctx.p < 2**38:
        pytest.skip("a reconstruction draws its residues by rejection from 63 bits: minutes for a prime this small")


# rational functions N/D with all terms of N and D in a box (D's first term 1):
# the balanced step with one and two registers of samples per lane
@pytest.mark.parametrize("nv,deg,TN,TD", [(3, 5, 30, 20), (2, 20, 60, 40)])
def test_reconstruct_rational(ctx, nv, deg, TN, TD):
    needs_draws(ctx)
    st, rnd = W.Stream(nv + deg, 1), random.Random(nv + deg)

    def function(T):
        e = W.distinct_monomials_box(st, T, nv, deg)
        e[0] = 0
        e = np.unique(e, axis=0)
        return e, rand_res(rnd, (e.shape[0],), ctx.p - 1) + np.uint64(1)
    (Ne, Nc), (De, Dc) = function(TN), function(TD)
    Dc[0] = 1
    degs = [deg] * nv
    (ne, nc), (de, dc), _ = ctx.reconstruct(nv, degs, 7, Ne, Nc, De, Dc, degD=degs)
    assert np.array_equal(ne, Ne) and np.array_equal(nc, Nc)
    assert np.array_equal(de, De) and np.array_equal(dc, Dc)


def test_reconstruct_poly(ctx):
    needs_draws(ctx)
    nv, T = 4, 2500
    e = W.distinct_monomials_box(W.Stream(3, 1), T, nv, 12)
    e = e[np.lexsort(e.T[::-1])]
    c = rand_res(random.Random(3), (T,), ctx.p - 1) + np.uint64(1)
    (ge, gc), _, _ = ctx.reconstruct(nv, [12] * nv, 5, e, c)
    assert np.array_equal(ge, e) and np.array_equal(gc, c)

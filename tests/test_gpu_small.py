"""GPU parity: entries solved in one launch (up to 256 unknowns and 32 samples)
at the edges of their roots (32 a CTA), k-blocks (8) and columns, alone and
beside larger entries, against the oracle."""
import random

import numpy as np
import pytest

from paper_2505_24256_gb300 import workloads as W
from tests.gpuutil import d8, d64, h64, rand_nodes, rand_res, zeros8, zeros64
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


def step(ctx, seed, T, S, k, maxexp, offset):
    """Descriptor, output buffers and the oracle's inputs of one step with random right-hand sides."""
    rnd = random.Random(seed)
    nv = k + 2                                    # the last variable is not touched
    skel = np.zeros((T, nv), dtype=np.uint8)
    if k:
        skel[:, :k] = W.distinct_monomials_box(W.Stream(seed, 1), T, k, maxexp)
    skel[:, k + 1] = 7
    y, cs = [rnd.randrange(1, P63) for _ in range(k)], rnd.sample(range(1, P63), S)
    b = rand_res(rnd, (S, T), P63)
    b[rnd.randrange(S)] = 0
    oe, oc, on = zeros8(T * S, nv), zeros64(T * S), zeros64(1)
    keep = [d8(skel), d64(y or [0]), d64(cs), d64(b)]
    d = dict(skel=ctx.poly(nv, T, keep[0]), newvar=k, S=S, offset=offset, y=keep[1], samples=keep[2], probes=keep[3],
             ldb=T, out_exps=oe, out_coef=oc, out_cap=T * S, out_count=on)
    return d, keep, (skel, k, y, cs, b, offset)


def check(orc, d, ref):
    skel, k, y, cs, b, offset = ref
    we, wc = orc.zippel_step(skel, k, y, cs, b, offset=offset)
    n = int(d["out_count"][0])
    assert n == we.shape[0]
    assert np.array_equal(d["out_exps"][:n].cpu().numpy(), we) and np.array_equal(h64(d["out_coef"][:n]), wc)


@pytest.mark.parametrize("T,k,maxexp", [(1, 0, 0), (1, 3, 9), (2, 1, 200), (7, 1, 255), (8, 2, 40), (9, 2, 40),
                                        (31, 3, 255), (32, 1, 255), (33, 6, 3), (64, 2, 9), (65, 2, 20), (200, 2, 20),
                                        (255, 5, 20), (256, 1, 255), (257, 2, 30)])
@pytest.mark.parametrize("S,offset", [(1, 1), (4, 0), (11, 1), (32, 0), (33, 0)])
def test_small_step(ctx, orc, T, k, maxexp, S, offset):
    d, keep, ref = step(ctx, 1000 * T + S, T, S, k, maxexp, offset)
    ctx.zippel_step_batched([d])
    check(orc, d, ref)


def test_small_among_others(ctx, orc):
    sizes = [(20, 3), (1, 1), (300, 5), (256, 21), (2500, 21), (40, 40), (4100, 6), (66, 11)]
    made = [step(ctx, 77 + i, T, S, 4, 20, i % 2) for i, (T, S) in enumerate(sizes)]
    for _ in range(2):
        ctx.zippel_step_batched([m[0] for m in made])
        for d, _, ref in made:
            check(orc, d, ref)
            d["out_coef"].zero_()


@pytest.mark.parametrize("sizes", [[(1, 1), (33, 4), (256, 32), (97, 13)], [(200, 3), (700, 5), (5, 33), (64, 1)]])
def test_small_systems(ctx, orc, sizes):
    rnd = random.Random(len(sizes) + sizes[0][0])
    for offset in (0, 1):
        sysv, refs = [], []
        for T, S in sizes:
            v, b = rand_nodes(rnd, T, P63), rand_res(rnd, (S, T), P63)
            c = zeros64(S, T)
            sysv.append(dict(T=T, S=S, offset=offset, v=d64(v), b=d64(b), ldb=T, c=c, ldc=T))
            refs.append((v, b))
        ctx.vandermonde_solve(sysv)
        for s, (v, b) in zip(sysv, refs):
            assert np.array_equal(h64(s["c"]), orc.tvandermonde_solve(v, b, offset=offset))


@pytest.mark.parametrize("T", [2, 33, 200])
def test_small_failures(ctx, orc, T):
    from paper_2505_24256_gb300 import zr

    rnd = random.Random(T)
    v, b = rand_nodes(rnd, T, P63), rand_res(rnd, (2, T), P63)

    def status(v, offset):
        c = zeros64(2, T)
        with pytest.raises(zr.ZrError) as e:
            ctx.vandermonde_solve([dict(T=T, S=2, offset=offset, v=d64(v), b=d64(b), ldb=T, c=c, ldc=T)])
        return e.value.status

    w = v.copy()
    w[T - 1] = w[0]
    assert status(w, 0) == zr.SINGULAR               # equal nodes
    w = v.copy()
    w[T // 2] = 0
    assert status(w, 1) == zr.SINGULAR               # a zero node with exponents from 1
    d, keep, ref = step(ctx, 5 * T, T, 3, 2, 20, 0)
    keep[2][1] = keep[2][0]
    with pytest.raises(zr.ZrError) as e:
        ctx.zippel_step_batched([d])                 # equal samples
    assert e.value.status == zr.SINGULAR
    d, keep, ref = step(ctx, 5 * T, T, 3, 2, 20, 0)
    ctx.zippel_step_batched([d])
    check(orc, d, ref)


def test_small_step_is_one_launch(ctx, orc):
    from paper_2505_24256_gb300 import zr

    d, keep, ref = step(ctx, 9, 256, 21, 5, 20, 0)
    before = zr.launch_count()
    ctx.zippel_step_batched([d])
    assert zr.launch_count() - before == 1
    check(orc, d, ref)

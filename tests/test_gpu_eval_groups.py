"""GPU parity: the merged weights of groups of several terms, a block and a thread
per group, for each of the evaluators that read them, and the evaluation of few
terms at many points, against the oracle."""
import numpy as np
import pytest

from paper_2505_24256_gb300 import workloads as W
from tests.gpuutil import d8, d64, h64, zeros64
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


# a block per group at the two edges of its rule (8 terms on average, 80 n
# groups), more groups than blocks, and a thread per entry beyond them; the
# ring kernel, the tensor cores (T (S + 4) T >= 3.3e7), the tree
@pytest.mark.parametrize("G,n", [(640, 8), (650, 8), (700, 7), (1500, 20), (2560, 32), (2600, 32), (33, 255)])
@pytest.mark.parametrize("S,T,method", [(1, 40, 0), (3, 3300, 0), (9, 50, 2)])
def test_weights(ctx, orc, G, n, S, T, method):
    nv, k = 6, 5
    code = np.arange(G)
    exps = np.zeros((G * n, nv), dtype=np.uint8)
    for m in range(k):
        exps[:, m] = np.repeat((code // 7**m) % 7, n)
    exps[:, k] = np.tile(np.arange(n), G)
    st = W.Stream(G + n, 3)
    order = np.argsort(st.raw(G * n))
    exps = np.ascontiguousarray(exps[order])
    coef, y, cs, z = st.residues(G * n), st.residues(k), st.residues(S), st.residues(nv)
    out = zeros64(S, T)
    ke, kc, ky, kcs, kz = d8(exps), d64(coef), d64(y), d64(cs), d64(z)
    ctx.solve_method(method)
    try:
        ctx.zippel_probes(ctx.poly(nv, G * n, ke, kc), k, ky, S, kcs, kz, T, 1, out, T)
    finally:
        ctx.solve_method(0)
    sidx, iidx = st.below(40, S), np.concatenate([[0, T - 1], st.below(38, T)])
    want = orc.zippel_probes_sampled(exps, coef, k, y, cs, z, sidx, iidx, offset=1)
    assert np.array_equal(h64(out)[sidx, iidx], want)


@pytest.mark.parametrize("Tf", [0, 1, 31, 32, 33])
@pytest.mark.parametrize("nv,maxexp,npts", [(1, 255, 1217), (5, 20, 1216), (5, 255, 2003), (64, 3, 1500)])
def test_few_terms_at_many_points(ctx, orc, Tf, nv, maxexp, npts):
    exps = W.Stream(Tf, 1).below(Tf * nv, maxexp + 1).reshape(Tf, nv).astype(np.uint8)
    coef, pts = W.Stream(Tf, 2).residues(Tf), W.Stream(npts, 3).residues(npts * nv).reshape(npts, nv)
    out = zeros64(npts)
    ke, kc, kp = d8(exps), d64(coef), d64(pts)
    ctx.eval_points(ctx.poly(nv, Tf, ke, kc), npts, kp, out)
    assert np.array_equal(h64(out), orc.eval_points(exps, coef, pts))

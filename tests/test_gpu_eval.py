"""GPU parity: the evaluator's grouping (few large groups, single-term groups,
one and several column blocks) and the evaluation at explicit points (one CTA
and a cluster per point), against the oracle."""
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


def function(seed, Tf, nv, maxexp):
    st = W.Stream(seed, 1)
    return W.distinct_monomials_box(st, Tf, nv, maxexp), st.residues(Tf)


@pytest.mark.parametrize("Tf,nv,k,maxexp", [(1, 2, 1, 3), (700, 4, 1, 9), (700, 4, 0, 9), (900, 4, 3, 9),
                                            (2100, 5, 1, 6), (257, 3, 2, 255)])
@pytest.mark.parametrize("S,T,offset", [(1, 1, 0), (33, 40, 1), (70, 31, 0)])
def test_probes_groups(ctx, orc, Tf, nv, k, maxexp, S, T, offset):
    exps, coef = function(7 * Tf + k, Tf, nv, maxexp)
    st = W.Stream(Tf + S, 2)
    y, cs, z = st.residues(max(k, 1)), st.residues(S), st.residues(nv)
    out = zeros64(S, T)
    ke, kc, ky, kcs, kz = d8(exps), d64(coef), d64(y), d64(cs), d64(z)
    ctx.zippel_probes(ctx.poly(nv, Tf, ke, kc), k, ky, S, kcs, kz, T, offset, out, T)
    assert np.array_equal(h64(out), orc.zippel_probes(exps, coef, k, y[:k], cs, z, T, offset))


@pytest.mark.parametrize("Tf,nv,maxexp,npts", [(0, 2, 3, 5), (1, 1, 255, 3), (256, 3, 20, 2), (257, 3, 255, 2),
                                               (3000, 5, 20, 33), (3000, 5, 20, 300), (520, 64, 3, 7)])
def test_eval_points_clusters(ctx, orc, Tf, nv, maxexp, npts):
    exps, coef = function(Tf + nv, Tf, nv, maxexp) if nv < 9 else (
        W.Stream(3, 1).below(Tf * nv, maxexp + 1).reshape(Tf, nv).astype(np.uint8), W.Stream(3, 2).residues(Tf))
    pts = W.Stream(npts, 3).residues(npts * nv).reshape(npts, nv)
    out = zeros64(npts)
    ke, kc, kp = d8(exps), d64(coef), d64(pts)
    ctx.eval_points(ctx.poly(nv, Tf, ke, kc), npts, kp, out)
    assert np.array_equal(h64(out), orc.eval_points(exps, coef, pts))

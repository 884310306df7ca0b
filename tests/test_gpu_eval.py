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


# the product on the tensor cores: S T Tf above its threshold, odd tiles of
# rows (128) and columns (32), k-steps (16 groups) and chunks (128), a single
# column, more than 64 columns, few groups
@pytest.mark.parametrize("Tf,nv,k,maxexp,S,T,offset", [(1500, 5, 4, 9, 33, 700, 1), (2600, 6, 5, 9, 1, 1601, 0),
                                                       (2600, 3, 1, 255, 21, 1000, 1), (2000, 5, 3, 9, 70, 300, 0),
                                                       (4097, 5, 4, 20, 11, 1409, 0)])
def test_probes_tensor_cores(ctx, orc, Tf, nv, k, maxexp, S, T, offset):
    test_probes_groups(ctx, orc, Tf, nv, k, maxexp, S, T, offset)


def test_probes_tensor_cores_extreme_digits(ctx, orc):
    """Anchor values and weights whose base-256 digits are all -128 or 127 but
    for the lowest and the top one: the antidiagonal sums come near their bound."""
    nv, k, T, S = 64, 63, 5000, 60
    low = sum(128 << (8 * i) for i in range(1, 7))
    y = np.array([(P63 - low + (5 + t)) % P63 if t % 2 else sum(127 << (8 * i) for i in range(1, 7)) + t
                  for t in range(k)], dtype=np.uint64)
    exps = np.zeros((k, nv), dtype=np.uint8)
    exps[np.arange(k), np.arange(k)] = 1
    coef = np.array([P63 - low - 128 if t % 2 else P63 - low + 127 for t in range(k)], dtype=np.uint64)
    cs = np.concatenate([[1], W.Stream(5, 1).distinct_residues(S - 1, avoid=[1])]).astype(np.uint64)
    out = zeros64(S, T)
    ke, kc, ky, kcs = d8(exps), d64(coef), d64(y), d64(cs)
    ctx.zippel_probes(ctx.poly(nv, k, ke, kc), k, ky, S, kcs, None, T, 0, out, T)
    assert np.array_equal(h64(out), orc.zippel_probes(exps, coef, k, y, cs, np.zeros(nv, np.uint64), T))


def test_probes_tensor_cores_long_sums(ctx, orc):
    """More than 128 chunks of 128 groups in one unit: the words' carries run."""
    Tf, nv, k, S, T = 1 << 17, 6, 5, 64, 3000
    exps, coef = function(91, Tf, nv, 20)
    st = W.Stream(92, 2)
    y, cs, z = st.residues(k), st.residues(S), st.residues(nv)
    out = zeros64(S, T)
    ke, kc, ky, kcs, kz = d8(exps), d64(coef), d64(y), d64(cs), d64(z)
    ctx.solve_method(1)
    ctx.zippel_probes(ctx.poly(nv, Tf, ke, kc), k, ky, S, kcs, kz, T, 0, out, T)
    ctx.solve_method(0)
    sidx, iidx = st.below(40, S).astype(np.int64), st.below(40, T).astype(np.int64)
    want = orc.zippel_probes_sampled(exps, coef, k, y, cs, z, sidx, iidx)
    assert np.array_equal(h64(out)[sidx, iidx], want)


def test_probes_many_groups_of_several_terms(ctx, orc):
    test_probes_groups(ctx, orc, 90000, 5, 4, 9, 8, 31, 1)

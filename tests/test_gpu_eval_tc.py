"""GPU parity of the evaluator's product on the tensor cores, at the edges of its
tiles and sums, against the oracle."""
import numpy as np
import pytest

from paper_2505_24256_gb300 import workloads as W
from tests.gpuutil import d8, d64, h64, zeros64
from tests.pyref import P63

pytestmark = pytest.mark.gpu


@pytest.fixture
def ctx():
    import __graft_entry__ as ge
    from paper_2505_24256_gb300 import zr

    ge.build()
    c = zr.Context(P63)                            # a workspace of its own
    yield c
    c.close()


def probes(ctx, exps, coef, k, y, cs, z, T, offset=0):
    S, nv = len(cs), exps.shape[1]
    out = zeros64(S, T)
    ke, kc, ky, kcs, kz = d8(exps), d64(coef), d64(y), d64(cs), d64(z)
    ctx.zippel_probes(ctx.poly(nv, exps.shape[0], ke, kc), k, ky, S, kcs, kz, T, offset, out, T)
    return h64(out)


@pytest.mark.parametrize("T,Tf,S,offset", [(2200000, 8192, 1, 1), (1200000, 4100, 3, 0)])
def test_scratch_does_not_grow_with_the_probes(ctx, orc, T, Tf, S, offset):
    """More probes than a slab of giant steps holds (2^25 words, a row of Tf for
    128 probes): 1.1 GB of them together in the first case, three slabs."""
    nv, k = 5, 4
    exps, coef = W.distinct_monomials_box(W.Stream(Tf, 1), Tf, nv, 20), W.Stream(Tf, 2).residues(Tf)
    st = W.Stream(Tf + S, 2)
    y, cs, z = st.residues(k), st.residues(S), st.residues(nv)
    out = probes(ctx, exps, coef, k, y, cs, z, T, offset)
    assert ctx.workspace_bytes() < 450 << 20
    slab = 128 * ((1 << 25) // (-(-Tf // 16) * 16))
    edges = [i + d for i in range(0, T, slab) for d in (-1, 0, 1, 127, 128) if 0 <= i + d < T] + [T - 1]
    iidx = np.array(edges + st.below(30, T).tolist(), dtype=np.int64)
    for s in range(S):
        sidx = np.full(len(iidx), s)
        want = orc.zippel_probes_sampled(exps, coef, k, y, cs, z, sidx, iidx, offset=offset)
        assert np.array_equal(out[s, iidx], want)


@pytest.mark.parametrize("G,terms,T,S,tree", [((1 << 18) + 3, 1, 4096, 1, True), (70001, 4, 4099, 2, True),
                                              (4100, 64, 5000, 3, False)])
def test_many_terms_take_the_tree_by_their_groups(ctx, orc, G, terms, T, S, tree):
    """More terms than the tensor cores take: the transposed tree for enough
    groups, the integer kernel for few."""
    nv, k = 6, 5
    exps = np.zeros((G * terms, nv), dtype=np.uint8)
    code = np.arange(G)
    for m in range(k):
        exps[:, m] = np.repeat((code // 21**m) % 21, terms)
    exps[:, k] = np.tile(np.arange(terms), G)
    st = W.Stream(G, 3)
    coef, y, cs, z = st.residues(G * terms), st.residues(k), st.residues(S), st.residues(nv)
    ctx.profile(True)
    out = probes(ctx, exps, coef, k, y, cs, z, T)
    launches = ctx.profile_query("ntt")[1]
    ctx.profile(False)
    assert (launches > 0) == tree
    sidx, iidx = st.below(24, S), np.concatenate([[0, T - 1], st.below(22, T)])
    want = orc.zippel_probes_sampled(exps, coef, k, y, cs, z, sidx, iidx)
    assert np.array_equal(out[sidx, iidx], want)

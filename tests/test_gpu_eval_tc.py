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


# odd tiles of rows (128) and columns (32), k-steps (16 groups) and chunks (128);
# a single column, more than 64 and all 256; few groups and a single one
@pytest.mark.parametrize("Tf,nv,k,maxexp,S,T,offset", [(1500, 5, 4, 9, 33, 1100, 1), (2600, 6, 5, 9, 1, 2700, 0),
                                                       (2600, 3, 1, 255, 21, 1200, 1), (2000, 5, 3, 9, 70, 700, 0),
                                                       (4097, 5, 4, 20, 11, 1500, 0), (2000, 4, 0, 9, 60, 800, 1),
                                                       (401, 5, 4, 9, 256, 361, 0)])
def test_edges(ctx, orc, Tf, nv, k, maxexp, S, T, offset):
    assert ctx.probe_plan(T, Tf, S)[0] == ctx.PROBE_TC
    exps, coef = W.distinct_monomials_box(W.Stream(Tf, 1), Tf, nv, maxexp), W.Stream(Tf, 2).residues(Tf)
    st = W.Stream(Tf + S, 2)
    y, cs, z = st.residues(max(k, 1)), st.residues(S), st.residues(nv)
    want = orc.zippel_probes(exps, coef, k, y[:k], cs, z, T, offset)
    assert np.array_equal(probes(ctx, exps, coef, k, y, cs, z, T, offset), want)


def digits(x):
    """Balanced base-256 digits of the centred residue."""
    x = x - P63 if x > P63 >> 1 else x
    return [b - 128 for b in ((x + 0x8080808080808080) % 2**64).to_bytes(8, "little")]


def test_sums_near_their_bound(ctx, orc):
    """One chunk of 124 groups whose anchor values and weights have digits of -128
    and -127 but for the lowest and the top ones: the antidiagonal sums of the rows
    i = 1 come to 0.72 of the 2^24 up to which fp32 holds every integer."""
    nv, k, T, S = 64, 63, 4200, 60
    low = sum(128 << (8 * i) for i in range(1, 7))
    y = [P63 - low - 128 + a for a in range(62)] + [P63 - 1]
    exps = np.zeros((124, nv), dtype=np.uint8)
    for g in range(124):                           # y_a and -y_a
        exps[g, g // 2], exps[g, 62], exps[g, 63] = 1, g % 2, 1
    w = P63 - low - 128 - (63 << 56)
    sums = [0] * 15
    for g in range(124):
        for i, a in enumerate(digits(P63 - y[g // 2] if g % 2 else y[g // 2])):
            for j, b in enumerate(digits(w)):
                sums[i + j] += a * b
    largest = max(map(abs, sums)) / 2**24
    print("largest antidiagonal sum / 2^24:", largest)
    assert 0.7 < largest < 1
    coef = np.full(124, w, dtype=np.uint64)
    cs = np.concatenate([[1, P63 - 1], W.Stream(5, 1).distinct_residues(S - 2, avoid=[1, P63 - 1])]).astype(np.uint64)
    z = np.zeros(nv, dtype=np.uint64)
    assert ctx.probe_plan(T, 124, S)[0] == ctx.PROBE_TC
    assert np.array_equal(probes(ctx, exps, coef, k, y, cs, z, T), orc.zippel_probes(exps, coef, k, y, cs, z, T))


def test_more_chunks_than_a_carry_holds(ctx, orc):
    """More than 128 chunks of 128 groups in one work unit: the words' carries run
    (128 tiles of rows and 38 columns make 152 units of one split)."""
    Tf, nv, k, S, T = 40000, 6, 5, 38, 16384
    exps, coef = W.distinct_monomials_box(W.Stream(91, 1), Tf, nv, 20), W.Stream(91, 2).residues(Tf)
    st = W.Stream(92, 2)
    y, cs, z = st.residues(k), st.residues(S), st.residues(nv)
    ctx.solve_method(1)
    method, splits = ctx.probe_plan(T, Tf, S)
    assert method == ctx.PROBE_TC and Tf // (128 * splits) > 128
    out = probes(ctx, exps, coef, k, y, cs, z, T)
    edges = [0, 1, 127, 128, 129, 8191, T - 129, T - 128, T - 1]
    sidx = np.concatenate([np.repeat([0, 31, 32, S - 1], len(edges)), st.below(200, S)])
    iidx = np.concatenate([np.tile(edges, 4), st.below(200, T)])
    assert np.array_equal(out[sidx, iidx], orc.zippel_probes_sampled(exps, coef, k, y, cs, z, sidx, iidx))

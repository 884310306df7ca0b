"""GPU parity: step graphs of few and of many small entries (one launch, the chain
of kernels), against the oracle; the autotuner at shapes of small entries."""
import pytest

from tests.pyref import P63
from tests.test_gpu_small import check, step

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__ as ge
    from paper_2505_24256_gb300 import zr

    ge.build()
    c = zr.Context(P63)
    yield c
    c.close()


# two waves of clusters at most, and more than that, on any GPU of up to 512 SMs
@pytest.mark.parametrize("n,sizes,one", [(6, [(20, 3), (256, 21), (66, 4)], True), (1, [(1, 1)], True),
                                         (1500, [(20, 3), (31, 2), (1, 4), (9, 1)], False),
                                         (200, [(200, 2), (256, 5), (17, 3)], False)])
def test_graph_of_small_entries(ctx, orc, n, sizes, one):
    made = [step(ctx, 50 + i, *sizes[i % len(sizes)], 3, 20, i % 2) for i in range(n)]
    g = ctx.step_graph([m[0] for m in made])
    for d, _, _ in made:
        d["out_count"].fill_(-1)
        d["out_coef"].zero_()
    g.launch()
    g.status()
    assert (g.kernels == 1) == one
    for d, _, ref in made:                       # (an entry of one sample is all zeros: step)
        check(orc, d, ref)
    g.close()


def test_autotuner_times_plans_at_small_shapes(ctx):
    """Every candidate plan is run (twice) by the kernels it plans, not by the
    single launch that a small entry is elsewhere."""
    from paper_2505_24256_gb300 import zr

    before = zr.launch_count()
    ctx.autotune_step(200, 11, budget=3)
    assert zr.launch_count() - before >= 3 * 2 * 5
    assert ctx.step_plan(200, 11)[0] > 0

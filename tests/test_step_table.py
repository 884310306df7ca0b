"""The packed descriptor tables hold the bytes of the C structures, whatever form the entries come in."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
zr = pytest.importorskip("paper_2505_24256_gb300.zr")

TENSOR = torch.zeros(4, dtype=torch.int64)
ARRAY = np.zeros(4, dtype=np.uint64)


@pytest.mark.parametrize("buf", [TENSOR, ARRAY, 0x7000_0000_1000, None], ids=["tensor", "array", "address", "none"])
@pytest.mark.parametrize("num", [0, 7, -1, 2**31 + 5, np.int64(9)], ids=str)
def test_packed_rows_equal_the_structures(buf, num):
    skel = zr.zr_poly(3, 5, 0x1000, 0x2000)
    p = zr._ptr(buf)
    step = dict(newvar=2, S=num, offset=num, y=buf, samples=buf, probes=buf, ldb=num, out_exps=buf, out_coef=buf,
                out_cap=num, out_count=buf)
    want = bytes(zr.zr_step_desc(skel, 2, num, num, 0, p, p, p, num, p, p, num, p))
    for form in (skel, (3, 5, 0x1000, 0x2000)):
        assert zr._step_table([dict(step, skel=form)] * 2) == want * 2
    bare = {k: v for k, v in step.items() if k != "offset"}
    assert zr._step_table([dict(bare, skel=skel)]) == bytes(
        zr.zr_step_desc(skel, 2, num, 0, 0, p, p, p, num, p, p, num, p))
    syst = dict(T=num, S=num, offset=num, v=buf, b=buf, ldb=num, c=buf, ldc=num)
    assert zr._vsys_table([syst, syst]) == bytes(zr.zr_vsys(num, num, num, p, p, num, p, num)) * 2


def test_empty_lists_and_wrong_types():
    assert zr._step_table([]) == b"" and zr._vsys_table([]) == b""
    with pytest.raises(TypeError):
        zr._vsys_table([dict(T=1.5, S=1, v=0, b=0, ldb=1, c=0, ldc=1)])

"""The tree-resident grower draws a node's tried features by four lanes (features 0-15 in the first
half of their keys, 16-31 in the second): the same forest as the level-synchronous kernels' draw,
byte for byte, with one feature, all but one and about a third tried, on both sides of the halves
and at the most features it takes."""
import numpy as np
import pytest

from paper_1811_00156_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1811_00156_gb300 import aiwcrf as A


@pytest.mark.parametrize("F", [2, 5, 16, 17, 31, 32])
@pytest.mark.parametrize("part", ["one", "third", "all-but-one"])
def test_draw_of_four_lanes(F, part):
    import __graft_entry__
    __graft_entry__.build()
    mtry = {"one": 1, "third": max(1, F // 3), "all-but-one": F - 1}[part]
    wl = synth.small_case(40 + F, 900, F, card=40)
    X, y = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (wl.X, wl.y))
    out = []
    for g in (A.GROWER_TREE, A.GROWER_LEVEL):
        A.aiwcrf_set_grower(g)
        try:
            f = A.aiwcrf_fit(A.params(5, mtry, 1), X, y)
        finally:
            A.aiwcrf_set_grower(A.GROWER_AUTO)
        st = f.stats()
        assert st.pop("grower") == g
        out.append((f.serialize(), st))
    assert out[0] == out[1]

"""The tree-resident grower with 32, 16 and 8 warps a tree (the choice follows the number of trees):
the same forest as the level-synchronous kernels, byte for byte, on both sides of each line."""
import numpy as np
import pytest

from paper_1811_00156_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1811_00156_gb300 import aiwcrf as A


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    yield
    A.aiwcrf_set_grower(A.GROWER_AUTO)


def fit(grower, wl, prm):
    A.aiwcrf_set_grower(grower)
    try:
        return A.aiwcrf_fit(prm, torch.from_numpy(wl.X).cuda(), torch.from_numpy(wl.y).cuda())
    finally:
        A.aiwcrf_set_grower(A.GROWER_AUTO)


WORKLOADS = {
    "small nodes only": lambda: synth.small_case(21, 30, 6, card=9),
    "one level of big nodes": lambda: synth.small_case(22, 70, 6, card=256),
    "many big nodes": lambda: synth.small_case(23, 2500, 12, card=200),
    "ties": lambda: synth.small_case(24, 900, 5, card=3, y_levels=2),
}


@pytest.mark.parametrize("T", [1, 152, 153, 304, 305])
@pytest.mark.parametrize("name", WORKLOADS)
def test_forest_does_not_depend_on_the_warps(name, T):
    wl = WORKLOADS[name]()
    prm = A.params(T, 4, 2, seed=5)
    a, b = fit(A.GROWER_TREE, wl, prm), fit(A.GROWER_LEVEL, wl, prm)
    assert a.serialize() == b.serialize()
    sa, sb = a.stats(), b.stats()
    assert sa.pop("grower") == A.GROWER_TREE and sb.pop("grower") == A.GROWER_LEVEL
    assert sa == sb


def test_a_background_fit_gives_the_same_forest():
    wl = WORKLOADS["many big nodes"]()
    assert fit(A.GROWER_TREE, wl, A.params(20, 4, 2, seed=5)).serialize() == \
        fit(A.GROWER_TREE, wl, A.params(20, 4, 2, seed=5, ctas_per_sm=1)).serialize()

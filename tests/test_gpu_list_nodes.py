"""Presorted lists at the node sizes where their kernels change form: a root of 33 entries (the
smallest that has lists), 128 and 129 (a step of the search), 1,024 and 1,025 (split by a warp or
by a CTA), 4,096 and 4,097 (searched by a warp or by a CTA), 131,073 (no room for the split's bit
set), with distinct values and with ties, more features than a warp's lanes, and targets of three
values. The forest is that of the histogram search, byte for byte, and so are the fit's
counters."""
import numpy as np
import pytest

from paper_1811_00156_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1811_00156_gb300 import aiwcrf as A

# rows, features, values per column, targets' levels, trees, mtry, min_node
CASES = [(n, 4, card, 50, 2, 3, 1)
         for n in (33, 128, 129, 1024, 1025, 4096, 4097) for card in (0, 60)]
CASES += [(1500, 40, 0, 50, 2, 33, 2), (2500, 128, 300, 50, 2, 128, 5), (5000, 3, 0, 1, 2, 3, 1),
          (131073, 3, 3000, 50, 2, 2, 20)]


@pytest.mark.parametrize("n,F,card,levels,T,mtry,min_node", CASES)
def test_lists_match_histograms_at_the_edges(n, F, card, levels, T, mtry, min_node):
    import __graft_entry__
    __graft_entry__.build()
    kw = dict(y_levels=levels)
    if card:
        kw["card"] = card
    wl = synth.small_case(100 + n % 97, n, F, **kw)
    X, y = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (wl.X, wl.y))
    out = []
    for g in (A.GROWER_LISTS, A.GROWER_LEVEL):
        for bootstrap in (False, True):
            A.aiwcrf_set_grower(g)
            try:
                f = A.aiwcrf_fit(A.params(T, mtry, min_node, 0, 156, bootstrap), X, y)
            finally:
                A.aiwcrf_set_grower(A.GROWER_AUTO)
            st = f.stats()
            assert st.pop("grower") == g
            out.append((f.serialize(), st))
    assert out[0] == out[2] and out[1] == out[3]

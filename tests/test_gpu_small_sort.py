"""The presort of columns that one CTA sorts (up to 8,192 rows; 2, 4 or 8 rows a thread) and of the
first ones past it: the trees of the fit are the oracle's, node by node, on columns with distinct
values and with ties."""
import numpy as np
import pytest

import oracle as O
from paper_1811_00156_gb300 import synth
from tests.forest_util import assert_tree_equal, gpu_tree

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1811_00156_gb300 import aiwcrf as A


@pytest.mark.parametrize("card", [None, 90])
@pytest.mark.parametrize("n", [1, 33, 1024, 2048, 2049, 4096, 4097, 8192, 8193])
def test_presort_at_the_edges(n, card):
    import __graft_entry__
    __graft_entry__.build()
    wl = synth.small_case(60 + n % 50, n, 3, card=card)
    f = A.aiwcrf_fit(A.params(2, 2, 20), *(torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (wl.X, wl.y)))
    ref = O.fit(wl.X, wl.y, 2, 2, 20, seed=156)
    dec = A.decode_forest(f.serialize())
    for k in range(2):
        assert_tree_equal(gpu_tree(dec, k), ref.tree(k), where=f"tree {k}")

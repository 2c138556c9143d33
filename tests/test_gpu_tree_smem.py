"""The tree-resident grower at the most shared memory it takes with 32 warps a tree: trees whose
arrays leave between nothing and a little more than its own variables free of the 227 KB a CTA can
have (about 6,900 entries with 256 values a column) are grown, the same as by the level-synchronous
kernels."""
import numpy as np
import pytest

from paper_1811_00156_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1811_00156_gb300 import aiwcrf as A


def arrays(n, warps=32, bins=256):
    up = lambda x: (x + 15) & ~15
    return 12 * n + 3 * up(2 * n) + up(n) + warps * bins * 12 + 2 * up(2 * (n // 33 + 1))


ROWS = [n for n in range(6000, 8000) if 232448 - 2200 < arrays(n) <= 232448 - 900][::10]


@pytest.mark.parametrize("n", ROWS)
def test_fits_up_to_the_shared_memory_of_a_cta(n):
    import __graft_entry__
    __graft_entry__.build()
    wl = synth.small_case(n, n, 4, card=256)
    assert max(len(np.unique(c)) for c in wl.X) == 256
    X, y = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (wl.X, wl.y))
    out = []
    for g in (A.GROWER_AUTO, A.GROWER_LEVEL):
        A.aiwcrf_set_grower(g)
        try:
            out.append(A.aiwcrf_fit(A.params(2, 2, 40, 0, 156, False), X, y).serialize())
        finally:
            A.aiwcrf_set_grower(A.GROWER_AUTO)
    assert out[0] == out[1]

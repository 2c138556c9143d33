"""Device selection on both sides of the lines between its kernels: few walks (tree-parallel), many
(the walk of predict on rows coded once per kernel), more than 64 devices (queries written out)."""
import numpy as np
import pytest

import oracle as O
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


def forests(F, card, T):
    wl = synth.small_case(3 * F + T, 300, F, card=card)
    wl.X[F - 2] = np.random.default_rng(1).integers(0, 15, 300)
    wl.X[F - 1] = np.random.default_rng(2).integers(0, 4, 300)
    gpu = A.aiwcrf_fit(A.params(T, F, 2, seed=9), torch.from_numpy(wl.X).cuda(), torch.from_numpy(wl.y).cuda())
    return gpu, O.fit(wl.X, wl.y, T, F, 2, seed=9)


def select(gpu, kf, size, ids, want_pred, ids_on_device=False):
    K = kf.shape[1]
    best = torch.full((K,), -9, dtype=torch.int32, device="cuda")
    pred = torch.full((K, len(ids)), -9, dtype=torch.int64, device="cuda") if want_pred else None
    A.aiwcrf_select_device(gpu, torch.from_numpy(np.ascontiguousarray(kf)).cuda(), size, ids, best, pred)
    torch.cuda.synchronize()
    return best.cpu().numpy(), None if pred is None else pred.cpu().numpy()


# card 40: one-byte codes; continuous: two-byte codes (300 values) and the 8-byte walk
@pytest.mark.parametrize("card", [40, None])
@pytest.mark.parametrize("F", [3, 5, 32])
@pytest.mark.parametrize("K,ids,size", [
    (1, [7], 0),                                            # tree-parallel
    (2185, list(range(14, -1, -1)), 3),                     # 2,097,600 walks at 64 trees: just past the line
    (2184, list(range(15)), 1),                             # ... and just before it
    (33, list(range(64)) , 2), (700, list(range(100, 36, -1)), 2),    # 64 devices, most of them unseen
    (32769, [3], 2),                                        # one device
    (40, list(range(65)), 1),                               # written out
    (2300, list(range(15)), -1),                            # a size class below every one
])
def test_selection_equals_the_oracle(card, F, K, ids, size):
    gpu, ref = forests(F, card, 64)
    kf = np.random.default_rng(K).normal(0.0, 3.0, (F - 2, K)).astype(np.float32)
    kf[0, :: 7] = np.nan
    rb, rp = ref.select_device(kf, size, ids)
    best, pred = select(gpu, kf, size, ids, True)
    assert np.array_equal(best, rb) and np.array_equal(pred.reshape(-1), np.asarray(rp).reshape(-1))
    assert np.array_equal(select(gpu, kf, size, ids, False)[0], rb)

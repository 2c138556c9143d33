"""Device selections just before and just past the lines between the tree-parallel kernel and the batch
walk: CTAs of 32 trees, few or many devices, batches that are sorted, several passes of devices."""
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


# card 40: one-byte codes; continuous: two-byte codes, whose batches are never sorted
@pytest.mark.parametrize("card", [40, None])
@pytest.mark.parametrize("T,D,K", [
    (1, 1, 2048), (1, 1, 2049), (33, 8, 1024), (33, 8, 1025),       # few devices: 2,048 CTAs
    (32, 9, 4096), (32, 9, 4097), (65, 15, 1365), (65, 15, 1366),   # 4,096
    (1, 17, 2730), (1, 17, 2731), (2, 64, 1638), (2, 64, 1639),     # two and four passes of devices
    (1, 15, 12288), (1, 15, 12289), (40, 64, 2457), (40, 64, 2458), # sorted: 12,288
    (1, 1, 70000),                                                  # few trees, many kernels
])
def test_selection_on_both_sides_of_the_lines(card, T, D, K):
    F = 5
    wl = synth.small_case(F + T, 300, F, card=card)
    wl.X[F - 2] = np.random.default_rng(1).integers(0, 64, 300)
    wl.X[F - 1] = np.random.default_rng(2).integers(0, 4, 300)
    gpu = A.aiwcrf_fit(A.params(T, F, 2, seed=9), torch.from_numpy(wl.X).cuda(), torch.from_numpy(wl.y).cuda())
    ref = O.fit(wl.X, wl.y, T, F, 2, seed=9)
    kf = np.random.default_rng(K).normal(0.0, 3.0, (F - 2, K)).astype(np.float32)
    ids = list(range(D))[::-1]
    best = torch.full((K,), -9, dtype=torch.int32, device="cuda")
    pred = torch.empty(K, D, dtype=torch.int64, device="cuda")
    A.aiwcrf_select_device(gpu, torch.from_numpy(kf).cuda(), 2, ids, best, pred)
    rb, rp = ref.select_device(kf, 2, ids)
    assert np.array_equal(pred.cpu().numpy(), rp) and np.array_equal(best.cpu().numpy(), rb)

"""Device ids of a selection: negative ones on every route, and page-locked ids that earlier work of
the call's stream writes."""
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


def forests(T=64):
    wl = synth.small_case(5, 300, 5, card=40)
    wl.X[3] = np.random.default_rng(1).integers(-4, 12, 300)
    wl.X[4] = np.random.default_rng(2).integers(0, 4, 300)
    gpu = A.aiwcrf_fit(A.params(T, 5, 2, seed=9), torch.from_numpy(wl.X).cuda(), torch.from_numpy(wl.y).cuda())
    return gpu, O.fit(wl.X, wl.y, T, 5, 2, seed=9)


def fastest(pred, ids):
    """The device of the smallest prediction, the lower id on a tie."""
    order = np.argsort(ids, kind="stable")
    return np.asarray(ids, np.int32)[order][np.argmin(np.asarray(pred)[:, order], axis=1)]


# few walks, many walks, more devices than travel with a launch
@pytest.mark.parametrize("K,ids", [(50, [-3, 5, -1, 2]), (20000, [-3, 5, -1, 2]), (40, list(range(-70, 5)))])
def test_negative_device_ids(K, ids):
    gpu, ref = forests()
    kf = np.random.default_rng(K).normal(0.0, 3.0, (3, K)).astype(np.float32)
    best = torch.full((K,), -9, dtype=torch.int32, device="cuda")
    pred = torch.empty(K, len(ids), dtype=torch.int64, device="cuda")
    A.aiwcrf_select_device(gpu, torch.from_numpy(kf).cuda(), 1, ids, best, pred)
    rp = ref.select_device(kf, 1, ids)[1]
    assert np.array_equal(pred.cpu().numpy(), rp)
    assert np.array_equal(best.cpu().numpy(), fastest(rp, ids))


@pytest.mark.parametrize("K", [3, 20000])
def test_page_locked_ids_are_read_in_stream_order(K):
    """Host inputs are copied on the call's stream: ids that the stream's earlier work writes into
    page-locked memory are the ones that count."""
    gpu, ref = forests()
    kf = np.random.default_rng(K).normal(0.0, 3.0, (3, K)).astype(np.float32)
    dk = torch.from_numpy(kf).cuda()
    old, new = [0, 1, 2, 3], [9, -2, 6, 4]
    ids = torch.tensor(old, dtype=torch.int32).pin_memory()
    dnew = torch.tensor(new, dtype=torch.int32, device="cuda")
    best = torch.full((K,), -9, dtype=torch.int32, device="cuda")
    pred = torch.empty(K, 4, dtype=torch.int64, device="cuda")
    big = torch.randn(4096, 4096, device="cuda")
    A.aiwcrf_select_device(gpu, dk, 1, old, best, pred)             # everything is loaded
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        for _ in range(20):                                         # some milliseconds before the ids are written
            big = big @ big * 1e-4
        ids.copy_(dnew, non_blocking=True)
        A.aiwcrf_select_device(gpu, dk, 1, ids.numpy(), best, pred)
    torch.cuda.synchronize()
    rp = ref.select_device(kf, 1, new)[1]
    assert np.array_equal(pred.cpu().numpy(), rp)
    assert np.array_equal(best.cpu().numpy(), fastest(rp, new))

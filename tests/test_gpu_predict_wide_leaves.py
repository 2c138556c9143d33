"""The ensemble variance where its sum of squares needs more than 96 bits: many trees of the largest
targets, and a checkpoint's leaves beyond them, with the trees of a call split over CTAs."""
import struct

import numpy as np
import pytest

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


def stumps(thr, left, right):
    """A checkpoint of one split on feature 0 a tree: x <= thr gives left, else right."""
    T = len(thr)
    n = np.zeros((T, 4), np.uint64)
    mask = np.uint64((1 << 63) - 1)
    n[:, 0] = np.uint64(1 << 32) | np.asarray(thr, np.float32).view(np.uint32).astype(np.uint64)
    n[:, 1] = np.uint64(1 << 63) | (np.asarray(left, np.int64).view(np.uint64) & mask)
    n[:, 2] = np.uint64(1 << 63) | (np.asarray(right, np.int64).view(np.uint64) & mask)
    n[:, 3] = np.uint64(1 << 63)
    head = b"AIWCRF01" + struct.pack("<IIqq", 1, 1, T, 4 * T)
    return A.aiwcrf_forest_deserialize(head + (4 * np.arange(T + 1, dtype=np.int64)).tobytes() + n.tobytes())


# steps: distinct thresholds (over 255 of them: two-byte codes and the 8-byte walk)
@pytest.mark.parametrize("T,leaf,steps", [
    (1 << 16, 1 << 40, 7), (1 << 16, 1 << 40, 300), (1 << 17, 1 << 40, 7),       # the largest targets
    (16, 1 << 47, 7), (600, 1 << 56, 300),                                       # a checkpoint's larger leaves
])
@pytest.mark.parametrize("Q", [5, 700])
def test_variance_keeps_all_its_bits(T, leaf, steps, Q):
    rng = np.random.default_rng(T)
    thr = (np.arange(T) % steps).astype(np.float32)
    left = leaf - rng.integers(0, 3, T)
    right = np.where(np.arange(T) % 2 == 0, -leaf, leaf).astype(np.int64)
    forest = stumps(thr, left, right)
    x = np.linspace(-1.0, steps, Q).astype(np.float32)              # from every left leaf to every right one
    out = torch.empty(Q, dtype=torch.int64, device="cuda")
    var = torch.empty(2 * Q, dtype=torch.int64, device="cuda")
    A.aiwcrf_predict(forest, torch.from_numpy(x[None]).cuda(), out, var)
    torch.cuda.synchronize()
    got, gv = out.cpu().numpy(), var.cpu().numpy().view(np.uint64)
    for q in {0, 1, Q // 2, Q - 2, Q - 1}:
        v = [int(a) for a in np.where(x[q] <= thr, left, right)]
        P = (sum(v) + (1 << 63)) % (1 << 64) - (1 << 63)                # the trees' sum is an int64
        V = (T * sum(a * a for a in v) - P * P) % (1 << 128)             # two words
        assert int(gv[2 * q]) | int(gv[2 * q + 1]) << 64 == V
        assert int(got[q]) == (2 * P + T) // (2 * T)

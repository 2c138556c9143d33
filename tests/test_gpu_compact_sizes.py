"""Compact forests (at most 255 values a column) around the sizes where their form or their walk changes:
trees that fit a shared-memory slot (12,288 nodes) or not, children as byte offsets (up to 16,384 nodes) or
as indices (up to 65,536), and past that the 8-byte walk."""
import struct

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


F = 6


def tree(nodes, rng, grid):
    """Feature (-1: leaf), left child, threshold and value of a complete tree of nodes - 1 nodes and a pad."""
    n = nodes - 1
    j = np.arange(nodes)
    split = 2 * j + 2 < n
    feat = np.where(split, rng.integers(0, F, nodes), -1)
    val = rng.integers(-(1 << 40), 1 << 40, nodes)
    val[n] = 0
    return feat, np.where(split, 2 * j + 1, 0), grid[rng.integers(0, grid.size, nodes)], val


def checkpoint(trees):
    words = []
    for feat, left, thr, val in trees:
        sp = feat.astype(np.int64).clip(0).astype(np.uint64) << np.uint64(56) | left.astype(np.uint64) << np.uint64(32)
        sp |= thr.view(np.uint32).astype(np.uint64)
        lf = np.uint64(1 << 63) | (val.astype(np.int64).view(np.uint64) & np.uint64((1 << 63) - 1))
        words.append(np.where(feat >= 0, sp, lf))
    off = np.concatenate([[0], np.cumsum([w.size for w in words])]).astype(np.int64)
    head = b"AIWCRF01" + struct.pack("<IIqq", 1, F, len(words), int(off[-1]))
    return A.aiwcrf_forest_deserialize(head + off.tobytes() + np.concatenate(words).astype(np.uint64).tobytes())


def leaves(trees, X):
    """(trees, queries) leaf values; a NaN goes right."""
    q = np.arange(X.shape[1])
    out = []
    for feat, left, thr, val in trees:
        j = np.zeros(q.size, np.int64)
        while True:
            f = feat[j]
            go = f >= 0
            if not go.any():
                break
            right = ~(X[f.clip(0), q] <= thr[j])
            j = np.where(go, left[j] + right, j)
        out.append(val[j])
    return np.stack(out)


def means(v):
    T = v.shape[0]
    return (2 * v.sum(0) + T) // (2 * T)                        # the sums of a few leaves stay far from 2^62


SIZES = [12288, 12290, 16384, 16386, 40002, 65536, 65538]


@pytest.mark.parametrize("nodes", SIZES)
@pytest.mark.parametrize("Q", [700, 70001])                     # in order, and sorted
def test_predict(nodes, Q):
    rng = np.random.default_rng(nodes)
    grid = np.sort(rng.normal(0.0, 2.0, 200)).astype(np.float32)
    trees = [tree(m, rng, grid) for m in (nodes, 64, 5000)]
    forest = checkpoint(trees)
    X = rng.normal(0.0, 2.0, (F, Q)).astype(np.float32)
    X[2, ::11] = np.nan
    v = leaves(trees, X)
    out, var = torch.empty(Q, dtype=torch.int64, device="cuda"), torch.empty(2 * Q, dtype=torch.int64, device="cuda")
    A.aiwcrf_predict(forest, torch.from_numpy(X).cuda(), out)
    assert np.array_equal(out.cpu().numpy(), means(v))
    out.fill_(-7)
    A.aiwcrf_predict(forest, torch.from_numpy(X).cuda(), out, var)
    assert np.array_equal(out.cpu().numpy(), means(v))
    w = var.cpu().numpy().view(np.uint64)
    for q in range(0, Q, Q // 300 + 1):
        a = [int(x) for x in v[:, q]]
        assert int(w[2 * q]) | int(w[2 * q + 1]) << 64 == 3 * sum(x * x for x in a) - sum(a) ** 2


@pytest.mark.parametrize("nodes", SIZES)
@pytest.mark.parametrize("K", [40, 30001])                      # tree-parallel, and the (sorted) batch walk
def test_selection(nodes, K):
    rng = np.random.default_rng(nodes)
    grid = np.sort(rng.normal(1.0, 2.0, 200)).astype(np.float32)
    trees = [tree(m, rng, grid) for m in (nodes, 64, 5000)]
    forest = checkpoint(trees)
    ids = [3, 0, -1]
    kf = rng.normal(0.0, 2.0, (F - 2, K)).astype(np.float32)
    X = np.concatenate([np.repeat(kf, 3, axis=1), np.tile(np.array(ids, np.float32), K)[None], np.full((1, 3 * K), 2.0, np.float32)])
    exp = means(leaves(trees, X)).reshape(K, 3)
    best, pred = torch.empty(K, dtype=torch.int32, device="cuda"), torch.empty(K, 3, dtype=torch.int64, device="cuda")
    A.aiwcrf_select_device(forest, torch.from_numpy(kf).cuda(), 2, ids, best, pred)
    assert np.array_equal(pred.cpu().numpy(), exp)
    order = np.argsort(ids, kind="stable")
    assert np.array_equal(best.cpu().numpy(), np.asarray(ids)[order][np.argmin(exp[:, order], axis=1)])


# rows of a column's 200 values, all different or in runs of four: trees of more nodes than a slot holds, and of more
# than byte offsets reach
@pytest.mark.parametrize("distinct,runs,lo,hi", [(11000, 1, 12288, 16384), (20000, 1, 16384, 65536), (7000, 4, 12288, 16384),
                                                 (9500, 4, 16384, 65536)])
def test_fit_and_out_of_bag(distinct, runs, lo, hi):
    wl = synth.small_case(distinct, distinct, F, card=200)
    X, y = np.ascontiguousarray(np.repeat(wl.X, runs, axis=1)), np.repeat(wl.y, runs)
    y = np.ascontiguousarray(y + np.arange(y.size) % 7 * 1000)
    forest = A.aiwcrf_fit(A.params(3, 3, 1, seed=9), torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda())
    off = np.diff(A.decode_forest(forest.serialize())["tree_off"])
    assert lo < off.max() <= hi
    ref = O.fit(X, y, 3, 3, 1, seed=9)
    s = torch.empty(y.size, dtype=torch.int64, device="cuda")
    c = torch.empty(y.size, dtype=torch.int32, device="cuda")
    A.aiwcrf_oob(forest, torch.from_numpy(X).cuda(), s, c)
    rs, rc = ref.oob(X)
    assert np.array_equal(s.cpu().numpy(), rs) and np.array_equal(c.cpu().numpy(), rc)
    Xq = torch.from_numpy(synth.small_case(5, 3000, F, card=200).X).cuda()
    exp = ref.predict(Xq.cpu().numpy())[0]
    for f in (forest, A.aiwcrf_forest_deserialize(forest.serialize())):
        out = torch.empty(3000, dtype=torch.int64, device="cuda")
        A.aiwcrf_predict(f, Xq, out)
        assert np.array_equal(out.cpu().numpy(), exp)

"""Predict with a call's trees split over CTAs: tile edges of the query count, one to many trees,
mean and variance, both walks, against the oracle and against the call's own slices."""
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


def predict(forest, Xq, var):
    X = torch.from_numpy(np.ascontiguousarray(Xq)).cuda()
    Q = X.shape[1]
    out = torch.empty(Q, dtype=torch.int64, device="cuda")
    ov = torch.empty(2 * Q, dtype=torch.int64, device="cuda") if var else None
    A.aiwcrf_predict(forest, X, out, ov)
    torch.cuda.synchronize()
    return out.cpu().numpy(), None if ov is None else ov.cpu().numpy().view(np.uint64)


def case(card, n, T):
    wl = synth.small_case(31 + T, n, 32, card=card)
    forest = A.aiwcrf_fit(A.params(T, 10, 2, seed=9), torch.from_numpy(wl.X).cuda(), torch.from_numpy(wl.y).cuda())
    return wl, forest


# card 40: one-byte codes and the compact walk; continuous columns of 300 rows: two-byte codes
@pytest.mark.parametrize("card,n", [(40, 300), (None, 300)])
@pytest.mark.parametrize("T", [1, 2, 37])
@pytest.mark.parametrize("Q", [1, 511, 512, 513, 1537])
def test_split_predict_equals_the_oracle(card, n, T, Q):
    wl, forest = case(card, n, T)
    ref = O.fit(wl.X, wl.y, T, 10, 2, seed=9)
    Xq = synth.small_case(5, Q, 32, card=card).X
    got, var = predict(forest, Xq, True)
    exp, _, ev = ref.predict(Xq, want_var=True)
    assert np.array_equal(got, exp)
    assert [int(var[2 * q]) | (int(var[2 * q + 1]) << 64) for q in range(Q)] == [int(v) for v in ev]


@pytest.mark.parametrize("var", [False, True])
def test_a_large_split_batch_equals_its_slices(var):
    """More tiles than the chip holds CTAs, with several parts each; slices of a thousand queries run
    with one tree per part, and the first of them against the oracle."""
    wl, forest = case(40, 300, 96)
    Q = 600_001
    Xq = synth.small_case(6, Q, 32, card=40).X
    got, gv = predict(forest, Xq, var)
    ref = O.fit(wl.X, wl.y, 96, 10, 2, seed=9)
    for a in [0, 65_536, 300_000, Q - 1000]:
        s, sv = predict(forest, Xq[:, a:a + 1000], var)
        assert np.array_equal(got[a:a + 1000], s)
        if var:
            assert np.array_equal(gv[2 * a:2 * (a + 1000)], sv)
    assert np.array_equal(got[:1000], ref.predict(Xq[:, :1000])[0])


# card 40 compact, continuous: the 8-byte walk; runs of alike rows as repeated measurements make them:
# a tile of 512 rows holds at most 128 different ones (so they alone are walked) from 4 in a row on
@pytest.mark.parametrize("card,runs", [(40, 1), (40, 3), (40, 4), (40, 50), (None, 3)])
@pytest.mark.parametrize("n,T", [(1, 3), (31, 1), (511, 2), (512, 37), (513, 37), (1537, 5), (1024, 400)])
def test_out_of_bag_sums_equal_the_oracle(card, runs, n, T):
    wl = synth.small_case(77 + n, (n + runs - 1) // runs, 32, card=card)
    X = np.ascontiguousarray(np.repeat(wl.X, runs, axis=1)[:, :n])
    y = np.ascontiguousarray(np.repeat(wl.y, runs)[:n])
    forest = A.aiwcrf_fit(A.params(T, 10, 2, seed=9), torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda())
    s = torch.full((n,), -7, dtype=torch.int64, device="cuda")
    c = torch.full((n,), -7, dtype=torch.int32, device="cuda")
    A.aiwcrf_oob(forest, torch.from_numpy(X).cuda(), s, c)
    torch.cuda.synchronize()
    ref = O.fit(X, y, T, 10, 2, seed=9)
    rs, rc = ref.oob(X)
    assert np.array_equal(s.cpu().numpy(), rs) and np.array_equal(c.cpu().numpy(), rc)
    pred = torch.empty(n, dtype=torch.int64, device="cuda")
    mse, rows = A.aiwcrf_oob_error(forest, torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda(), pred)
    rp, _, rrows = ref.oob_error(X, y)
    # the documented arithmetic: the exact sum of squares converted to double, divided once
    sq = sum((int(p) - int(v)) ** 2 for p, v, k in zip(rp, y, rc) if k > 0)
    exp = (float(sq >> 64) * 2.0 ** 64 + float(sq & (2 ** 64 - 1))) / rrows * 2.0 ** -64 if rrows else 0.0
    assert np.array_equal(pred.cpu().numpy(), rp) and mse == exp and rows == rrows

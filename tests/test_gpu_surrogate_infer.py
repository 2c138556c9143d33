"""The fused inference kernel over its input shapes: column counts at the edges of its groups of
eight inputs, several tiles per CTA with a ragged last one, and values that are no numbers."""
import numpy as np
import pytest

from oracle import mlp as M

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# the bound on the erf of the inference epilogues that tests/test_gpu_surrogate.py derives
ERF_INFER_ERR = 2e-6


@pytest.fixture(scope="module")
def A():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1811_00156_gb300 import aiwcrf
    return aiwcrf


def network(n_aiwc, n_dev, n_size, Q, seed):
    rng = np.random.default_rng(seed)
    P = rng.normal(0.0, 0.08, M.N_PARAMS).astype(np.float32)
    lg = (np.arange(n_aiwc) % 3 == 0).astype(np.uint8)
    X = rng.normal(0.0, 2.0, (n_aiwc + 2, Q)).astype(np.float32)
    X[:n_aiwc][lg == 1] = np.exp(np.abs(X[:n_aiwc][lg == 1])) + 0.5          # some below 1
    X[n_aiwc] = rng.integers(0, n_dev + 1, Q)                                # one value past the range
    X[n_aiwc + 1] = rng.integers(0, n_size, Q)
    mu = rng.normal(0.5, 0.2, n_aiwc).astype(np.float32)
    sd = rng.uniform(0.5, 2.5, n_aiwc).astype(np.float32)
    return P, X, mu, sd, lg


def predict(A, sg, X):
    out = torch.empty(X.shape[1], dtype=torch.float32, device="cuda")
    sg.predict(torch.from_numpy(np.ascontiguousarray(X)).cuda(), out)
    torch.cuda.synchronize()
    return out.cpu().numpy()


@pytest.mark.parametrize("n_aiwc,n_dev,n_size", [(1, 1, 1), (7, 2, 3), (8, 15, 4), (30, 15, 4), (33, 27, 4), (62, 1, 1)])
@pytest.mark.parametrize("Q", [129, 152 * 128 * 2 + 5])
def test_column_counts(A, n_aiwc, n_dev, n_size, Q):
    P, X, mu, sd, lg = network(n_aiwc, n_dev, n_size, Q, n_aiwc)
    sg = A.aiwcrf_surrogate_create(n_aiwc + 2, n_dev, n_size, P, mu, sd, lg)
    got = predict(A, sg, X)
    pick = np.unique(np.concatenate([np.arange(min(Q, 300)), np.arange(max(0, Q - 300), Q)]))
    ref, bound = M.forward_tolerance(P.astype(np.float64), X[:, pick], mu, sd, lg, n_dev, n_size, erf_err=ERF_INFER_ERR)
    assert np.all(np.abs(got[pick].astype(np.float64) - ref) <= bound)


def test_values_that_are_no_numbers(A):
    """A NaN or an infinite plain column makes its own query's output NaN and no other's; a NaN count
    column reads as 1 (log2 of the larger of it and 1), a NaN device as none."""
    P, X, mu, sd, lg = network(30, 15, 4, 700, 3)
    plain, count = int(np.flatnonzero(lg == 0)[0]), int(np.flatnonzero(lg == 1)[0])
    sg = A.aiwcrf_surrogate_create(32, 15, 4, P, mu, sd, lg)
    base = predict(A, sg, X)
    Y = X.copy()
    Y[plain, 5], Y[plain, 300], Y[plain, 301] = np.nan, np.inf, -np.inf
    got = predict(A, sg, Y)
    assert np.all(np.isnan(got[[5, 300, 301]]))
    rest = np.setdiff1d(np.arange(700), [5, 300, 301])
    assert np.array_equal(got[rest], base[rest])
    Y, Z = X.copy(), X.copy()
    Y[count, 9], Z[count, 9] = np.nan, 1.0
    Y[30, 10], Z[30, 10] = np.nan, 99.0
    assert np.array_equal(predict(A, sg, Y), predict(A, sg, Z))

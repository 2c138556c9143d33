"""The inference kernel's standardisation for deviations at the ends of FP32: subnormal ones and ones
whose reciprocal is subnormal, for values equal to the mean and away from it."""
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


@pytest.mark.parametrize("sd", [2.0 ** -149, 1e-40, 2.0 ** -126, 1.0, 2.0 ** 126, 2.0 ** 127])
def test_deviations_at_the_ends_of_fp32(A, sd):
    n_aiwc, Q = 9, 300
    rng = np.random.default_rng(5)
    P = rng.normal(0.0, 0.08, M.N_PARAMS).astype(np.float32)
    sd32 = np.full(n_aiwc, sd, np.float32)
    mu = np.zeros(n_aiwc, np.float32)
    lg = np.zeros(n_aiwc, np.uint8)
    k = rng.choice([0.0, 0.0, 1.0, -1.0, 1.5, -0.5], (n_aiwc, Q))            # zero: a value equal to the mean
    X = np.zeros((n_aiwc + 2, Q), np.float32)
    X[:n_aiwc] = (k * float(sd32[0])).astype(np.float32)
    X[n_aiwc], X[n_aiwc + 1] = rng.integers(0, 3, Q), rng.integers(0, 2, Q)
    sg = A.aiwcrf_surrogate_create(n_aiwc + 2, 3, 2, P, mu, sd32, lg)
    out = torch.empty(Q, dtype=torch.float32, device="cuda")
    sg.predict(torch.from_numpy(X).cuda(), out)
    ref, bound = M.forward_tolerance(P.astype(np.float64), X, mu, sd32, lg, 3, 2, erf_err=ERF_INFER_ERR)
    got = out.cpu().numpy().astype(np.float64)
    assert np.all(np.abs(got - ref) <= bound)

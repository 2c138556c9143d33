"""The training kernels' gradient and loss over their batch sizes: one tile of 128 rows, an odd number
of tiles, more tiles than the weight gradients have splits (64), one of them shorter; and a network
with fewer inputs. Every entry against the oracle within its running error analysis."""
import numpy as np
import pytest

from oracle import mlp as M
from tests.mlp_cases import model, violations

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def A():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1811_00156_gb300 import aiwcrf
    return aiwcrf


@pytest.mark.parametrize("n", [128, 384, 128 * 65, 128 * 129])
def test_gradient_at_batch_sizes(A, n):
    P, X, mu, sd, lg, y = model(n % 97, n)
    sg = A.aiwcrf_surrogate_create(32, 15, 4, P, mu, sd, lg)
    g = torch.full((M.N_PARAMS,), float("nan"), device="cuda")
    loss = torch.full((1,), float("nan"), device="cuda")
    sg.grad(torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda(), g, loss)
    torch.cuda.synchronize()
    rl, rg, lb, gb = M.grad_tolerance(P.astype(np.float64), X, mu, sd, lg, 15, 4, y.astype(np.float64))
    assert abs(float(loss.item()) - rl) <= lb
    v = violations(g.cpu().numpy(), rg, gb)
    assert all(c == 0 for c, _ in v.values()), v


def test_gradient_of_a_narrow_network(A):
    rng = np.random.default_rng(4)
    n, n_aiwc, n_dev, n_size = 256, 3, 5, 2
    P = rng.normal(0.0, 0.08, M.N_PARAMS).astype(np.float32)
    X = rng.normal(0.0, 1.0, (n_aiwc + 2, n)).astype(np.float32)
    X[n_aiwc], X[n_aiwc + 1] = rng.integers(0, n_dev, n), rng.integers(0, n_size, n)
    mu, sd, lg = np.zeros(n_aiwc, np.float32), np.ones(n_aiwc, np.float32), np.zeros(n_aiwc, np.uint8)
    y = rng.normal(-3.0, 1.0, n).astype(np.float32)
    sg = A.aiwcrf_surrogate_create(n_aiwc + 2, n_dev, n_size, P, mu, sd, lg)
    g, loss = torch.empty(M.N_PARAMS, device="cuda"), torch.empty(1, device="cuda")
    sg.grad(torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda(), g, loss)
    torch.cuda.synchronize()
    rl, rg, lb, gb = M.grad_tolerance(P.astype(np.float64), X, mu, sd, lg, n_dev, n_size, y.astype(np.float64))
    assert abs(float(loss.item()) - rl) <= lb
    v = violations(g.cpu().numpy(), rg, gb)
    assert all(c == 0 for c, _ in v.values()), v

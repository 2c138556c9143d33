"""The gradient of a batch of more tiles than a grid's second dimension holds. Every row is alike and every
value a small power of two, so that each sum is exact whatever its order."""
import numpy as np
import pytest

from oracle import mlp as M

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


@pytest.mark.parametrize("n", [1 << 14, 1 << 23])               # 128 and 65,536 tiles of 128 rows
def test_gradient_of_many_tiles(A, n):
    """With zero first-layer weights and biases both pre-activations are 0, GELU is 0 and GELU' 1/2: the output is b3,
    dz2 = d w3 / 2, dz1 = dz2 W2 / 2 with d = (b3 - y) / n."""
    free, _ = torch.cuda.mem_get_info()
    if free < 48 << 30:
        pytest.skip("needs 48 GB of device memory")
    w3 = 2.0 ** -(np.arange(M.HID) % 3)
    W2 = np.zeros((M.HID, M.HID))
    W2[np.arange(M.HID), (np.arange(M.HID) + 5) % M.HID] = 0.5
    P = np.zeros(M.N_PARAMS, np.float32)
    P[M.OW2:M.OB2], P[M.OW3:M.OB3], P[M.OB3] = W2.reshape(-1), w3, 1.5
    sg = A.aiwcrf_surrogate_create(3, 1, 1, P, np.zeros(1, np.float32), np.ones(1, np.float32), np.zeros(1, np.uint8))
    X = torch.zeros(3, n, device="cuda")                        # one column of value 2, device 0, size 0
    X[0] = 2.0
    y = torch.full((n,), 0.5, device="cuda")
    g = torch.full((M.N_PARAMS,), float("nan"), device="cuda")
    loss = torch.full((1,), float("nan"), device="cuda")
    sg.grad(X, y, g, loss)
    torch.cuda.synchronize()
    exp = np.zeros(M.N_PARAMS)                                  # b3 - y = 1
    dz2 = w3 / 2
    dz1 = dz2 @ W2 / 2
    W1 = np.zeros((M.HID, M.K_IN))
    W1[:, 0], W1[:, 1], W1[:, 2] = 2 * dz1, dz1, dz1
    exp[M.OW1:M.OB1], exp[M.OB1:M.OW2], exp[M.OB2:M.OW3], exp[M.OB3] = W1.reshape(-1), dz1, dz2, 1.0
    assert float(loss.item()) == 0.5 * n
    assert np.array_equal(g.cpu().numpy().astype(np.float64), exp)

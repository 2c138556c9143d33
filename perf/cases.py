"""The work a user of the library has it do, as cases that can be timed and compared.

A case is a dict of plain values; its "op" says which public call it makes (the C ABI of
include/aiwcrf.h through its ctypes binding). The data are the synthetic AIWC-shaped workloads of
synth.py: 37 kernels x 15 devices x 4 size classes, every cell run `reps` times. With rows =
"grid" a cell's runs share the kernel's feature vector (the features do not depend on the device or
the run); with rows = "per_row" every run has a vector of its own, so that no two rows are alike.

  select              device selection: n_kernels kernels x 15 devices on a resident forest
  predict             predicted times of n_queries fresh queries (var: and the ensemble variance)
  fit                 fit a forest and take its checkpoint to the host
  loko                leave-one-kernel-out: 37 forests in one batch, and their checkpoints
  oob                 out-of-bag error and predictions of the training rows (the tuner's objective)
  surrogate_predict   the distilled network's predictions of n_queries queries
  surrogate_grad      loss and gradient of one training batch of the network
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_1811_00156_gb300 import aiwcrf as A
from paper_1811_00156_gb300 import synth

CELLS = synth.N_KERNELS * synth.N_DEVICES * synth.N_SIZES     # 2,220 rows a repetition
F = synth.N_FEATURES
DEVICES = list(range(synth.N_DEVICES))
K_IN, HID = 64, 256                                           # the network's padded input and hidden widths
N_NET = HID * K_IN + HID + HID * HID + HID + HID + 1          # its parameters


def listed():
    return [
        # a scheduler asks for one kernel that is about to run: latency
        dict(name="select-1", op="select", n_kernels=1, reps=50, trees=500),
        # a full batch of the device-selection server
        dict(name="select-1024", op="select", n_kernels=1024, reps=50, trees=500),
        # the training table's own rows through a small forest (every row predicted once)
        dict(name="predict-2220", op="predict", n_queries=2220, var=False, rows="grid", reps=1, trees=128),
        # a middling, ragged batch with the ensemble variance beside the mean
        dict(name="predict-40001-var", op="predict", n_queries=40001, var=True, rows="grid", reps=50, trees=500),
        # the benchmark's batch: a sweep over a million hypothetical kernels
        dict(name="predict-1000000", op="predict", n_queries=1000000, var=False, rows="grid", reps=50, trees=500),
        # the plain forest of one measurement campaign without repeated runs
        dict(name="fit-2220", op="fit", rows="grid", reps=1, trees=128, mtry=10, min_node=5),
        # the benchmark's fit: 50 runs of every cell
        dict(name="fit-111000", op="fit", rows="grid", reps=50, trees=500, mtry=10, min_node=5),
        # the same table with a feature vector per run: wide ranks, nothing to group
        dict(name="fit-per-row", op="fit", rows="per_row", reps=50, trees=500, mtry=10, min_node=5),
        # cross-validation over kernels: 37 forests of uneven training sets
        dict(name="loko-256", op="loko", trees=256, mtry=10, min_node=5),
        # the error that parameter tuning asks for after every fit
        dict(name="oob-111000", op="oob", reps=50, trees=500, mtry=10, min_node=5),
        # the million-query sweep through the distilled network
        dict(name="surrogate-1000000", op="surrogate_predict", n_queries=1000000),
        # one step's gradient at the training batch size
        dict(name="surrogate-grad-4096", op="surrogate_grad", batch=4096),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    op = rng.choice(["select", "predict", "predict", "fit", "fit", "loko", "oob", "surrogate_predict",
                     "surrogate_grad"])
    trees = _log_int(rng, 16, 500)
    reps = _log_int(rng, 1, 50)
    if op == "select":      # up to a sweep of 65,536 kernels, where the query-parallel walk takes over
        return dict(op=op, n_kernels=_log_int(rng, 1, 65536), reps=reps, trees=trees)
    if op == "predict":
        rows = rng.choice(["grid", "grid", "grid", "per_row"])
        return dict(op=op, n_queries=_log_int(rng, 1, 1000000), var=rng.random() < 0.25, rows=rows,
                    reps=reps if rows == "grid" else _log_int(rng, 1, 5), trees=trees)
    if op == "fit":
        return dict(op=op, rows=rng.choice(["grid", "grid", "per_row"]), reps=reps, trees=trees,
                    mtry=rng.randint(4, 16), min_node=rng.randint(1, 20))
    if op == "loko":
        return dict(op=op, trees=_log_int(rng, 16, 256), mtry=rng.randint(4, 16), min_node=rng.randint(1, 20))
    if op == "oob":
        return dict(op=op, reps=reps, trees=trees, mtry=rng.randint(4, 16), min_node=rng.randint(1, 20))
    if op == "surrogate_predict":
        return dict(op=op, n_queries=_log_int(rng, 1, 1000000))
    return dict(op=op, batch=128 * _log_int(rng, 1, 128))


def _table(rows, reps, seed):
    """Training matrix and targets on the GPU."""
    make = synth.scaled_forest_workload if rows == "grid" else synth.per_row_forest_workload
    wl = make(seed, reps)
    return torch.from_numpy(wl.X).cuda(), torch.from_numpy(wl.y).cuda()


def _params(case, seed):
    return A.params(case["trees"], case.get("mtry", 10), case.get("min_node", 5), seed=seed & 0xFFFF)


def _queries(n, seed):
    return torch.from_numpy(synth.queries(n, seed)).cuda()


def _network(seed):
    """Host weights of the network (variance-preserving, random) and the standardisation of the
    AIWC columns: log2 of the counts, then mean and deviation of the columns' distributions."""
    g = torch.Generator().manual_seed(seed)
    w1 = torch.randn(HID, K_IN, generator=g) * (2.0 / (synth.N_AIWC + 2)) ** 0.5
    b1 = torch.randn(HID, generator=g) * 0.1
    w2 = torch.randn(HID, HID, generator=g) * (2.0 / HID) ** 0.5
    b2 = torch.randn(HID, generator=g) * 0.1
    w3 = torch.randn(HID, generator=g) * (1.0 / HID) ** 0.5
    b3 = torch.tensor([-3.0])
    P = torch.cat([t.reshape(-1) for t in (w1, b1, w2, b2, w3, b3)]).numpy()
    ln2, r12 = math.log(2.0), 12.0 ** 0.5
    mu = np.array([12.0 / ln2] * 10 + [16.0] * 8 + [0.5] * 6 + [14.0] * 6, np.float32)
    sd = np.array([3.0 / ln2] * 10 + [32.0 / r12] * 8 + [1.0 / r12] * 6 + [6.055] * 6, np.float32)
    lg = np.array([1] * 10 + [0] * 14 + [1] * 6, np.uint8)
    return P, mu, sd, lg


def _targets(n, seed):
    """log10 seconds of a batch, spread as the workloads' are."""
    g = torch.Generator().manual_seed(seed + 1)
    return torch.randn(n, generator=g) * 0.7 - 3.0


def prepare(case, seed):
    op = case["op"]
    st = dict(op=op)
    if op in ("select", "predict"):
        X, y = _table(case.get("rows", "grid"), case["reps"], seed)
        st["forest"] = A.aiwcrf_fit(_params(case, seed), X, y)
        if op == "select":
            K = case["n_kernels"]
            st["kfeat"] = torch.from_numpy(synth.queries(K, seed + 7)[: synth.N_AIWC].copy()).cuda()
            st["size"] = seed % synth.N_SIZES
            st["best"] = torch.empty(K, dtype=torch.int32, device="cuda")
            st["pred"] = torch.empty(K, len(DEVICES), dtype=torch.int64, device="cuda")
        else:
            n = case["n_queries"]
            st["Xq"] = _queries(n, seed + 7)
            st["pred"] = torch.empty(n, dtype=torch.int64, device="cuda")
            st["var"] = torch.empty(n, 2, dtype=torch.int64, device="cuda") if case["var"] else None
    elif op == "fit":
        st["X"], st["y"] = _table(case["rows"], case["reps"], seed)
        st["params"] = _params(case, seed)
        distinct = CELLS * (case["reps"] if case["rows"] == "per_row" else 1)
        st["blob"] = _blob(case["trees"], distinct)
    elif op == "loko":
        wl, folds = synth.loko_folds(seed)
        st["X"], st["y"] = torch.from_numpy(wl.X).cuda(), torch.from_numpy(wl.y).cuda()
        st["off"] = np.concatenate([[0], np.cumsum([tr.size for tr, _ in folds])]).astype(np.int64)
        st["rows"] = torch.from_numpy(np.concatenate([tr for tr, _ in folds]).astype(np.int32)).cuda()
        st["params"] = _params(case, seed)
        st["blobs"] = [_blob(case["trees"], CELLS) for _ in folds]
    elif op == "oob":
        st["X"], st["y"] = _table("grid", case["reps"], seed)
        st["forest"] = A.aiwcrf_fit(_params(case, seed), st["X"], st["y"])
        st["pred"] = torch.empty(CELLS * case["reps"], dtype=torch.int64, device="cuda")
    else:
        P, mu, sd, lg = _network(seed)
        st["net"] = A.aiwcrf_surrogate_create(F, synth.N_DEVICES, synth.N_SIZES, P, mu, sd, lg)
        n = case["n_queries"] if op == "surrogate_predict" else case["batch"]
        st["Xq"] = _queries(n, seed + 7)
        if op == "surrogate_predict":
            st["out"] = torch.empty(n, device="cuda")
        else:
            st["y"] = _targets(n, seed).cuda()
            st["grad"] = torch.empty(N_NET, device="cuda")
            st["loss"] = torch.empty(1, device="cuda")
    torch.cuda.synchronize()
    return st


def _blob(trees, distinct):
    """A pinned host buffer for a forest's checkpoint: a tree has at most 2 d + 1 nodes of 8 bytes,
    d its distinct in-bag rows: 0.632 of the distinct rows in expectation without repeated runs, all
    of them at most."""
    per_tree = 2 * distinct + 2 if distinct <= CELLS else int(1.3 * distinct) + 2
    return torch.zeros(4 + (trees + 1) + trees * per_tree, dtype=torch.int64, pin_memory=True)


def _checkpoint(forest, blob):
    """The forest's checkpoint, written to the head of the caller's buffer (the rest stays zero)."""
    need = ctypes.c_size_t()
    rc = A.load().aiwcrf_forest_serialize(forest.handle, blob.data_ptr(), 8 * blob.numel(), ctypes.byref(need))
    if rc != A.AIWCRF_OK:
        raise A.AiwcrfError(rc, A.load().aiwcrf_last_error().decode(errors="replace"))
    return blob


def run(st):
    op = st["op"]
    if op == "select":
        A.aiwcrf_select_device(st["forest"], st["kfeat"], st["size"], DEVICES, st["best"], st["pred"])
        return dict(best=st["best"], pred=st["pred"])
    if op == "predict":
        A.aiwcrf_predict(st["forest"], st["Xq"], st["pred"], st["var"])
        return dict(pred=st["pred"]) if st["var"] is None else dict(pred=st["pred"], var=st["var"])
    if op == "fit":
        st["forest"] = A.aiwcrf_fit(st["params"], st["X"], st["y"])
        return _checkpoint(st["forest"], st["blob"])
    if op == "loko":
        st["forests"] = A.aiwcrf_fit_subsets(st["params"], st["X"], st["y"], st["off"], st["rows"])
        return [_checkpoint(f, b) for f, b in zip(st["forests"], st["blobs"])]
    if op == "oob":
        mse, rows = A.aiwcrf_oob_error(st["forest"], st["X"], st["y"], st["pred"])
        return dict(mse=mse, rows=rows, pred=st["pred"])
    if op == "surrogate_predict":
        return st["net"].predict(st["Xq"], st["out"])
    st["net"].grad(st["Xq"], st["y"], st["grad"], st["loss"])
    return dict(grad=st["grad"], loss=st["loss"])


def _forest_bytes(case):
    """8 bytes a node of the checkpoint, 0.6 nodes a distinct row (measured at min_node 5: 0.41 without
    repeated runs, 0.74 with 50, 0.66 with 111,000 distinct rows)."""
    per_row = case.get("rows") == "per_row"
    return 8 * case["trees"] * 0.6 * CELLS * (case["reps"] if per_row else 1)


def work(case):
    op = case["op"]
    net = 2.0 * (K_IN * HID + HID * HID + HID)     # multiply-adds of one row forward, as 2 operations
    if op == "select":
        K = case["n_kernels"]
        return dict(bytes=4 * synth.N_AIWC * K + 4 * K + 8 * K * len(DEVICES), flops=0)
    if op == "predict":
        return dict(bytes=case["n_queries"] * (4 * F + 8 + (16 if case["var"] else 0)), flops=0)
    if op == "fit":
        return dict(bytes=CELLS * case["reps"] * (4 * F + 8) + _forest_bytes(case), flops=0)
    if op == "loko":
        one = dict(rows="grid", reps=1, trees=case["trees"])
        return dict(bytes=CELLS * (4 * F + 8) + synth.N_KERNELS * (4 * CELLS + _forest_bytes(one)), flops=0)
    if op == "oob":
        n = CELLS * case["reps"]
        return dict(bytes=n * (4 * F + 8 + 8) + n * case["trees"] / 8, flops=0)
    if op == "surrogate_predict":
        return dict(bytes=case["n_queries"] * (4 * F + 4) + 4 * N_NET, flops=case["n_queries"] * net)
    return dict(bytes=case["batch"] * (4 * F + 4) + 8 * N_NET, flops=case["batch"] * 3 * net)


def _encode64(X, mu, sd, lg):
    """(n, 64) network inputs in float64: standardised AIWC columns, one-hot device and size."""
    n = X.shape[1]
    x = X[: synth.N_AIWC].double()
    x = torch.where(torch.from_numpy(lg).bool().to(X.device)[:, None], torch.log2(x.clamp_min(1.0)), x)
    x = (x - torch.from_numpy(mu).double().to(X.device)[:, None]) / torch.from_numpy(sd).double().to(X.device)[:, None]
    out = torch.zeros(n, K_IN, dtype=torch.float64, device=X.device)
    out[:, : synth.N_AIWC] = x.T
    rows = torch.arange(n, device=X.device)
    out[rows, synth.N_AIWC + X[synth.COL_DEVICE].long()] = 1.0
    out[rows, synth.N_AIWC + synth.N_DEVICES + X[synth.COL_SIZE].long()] = 1.0
    return out


def exact(case, seed):
    """The network in float64. The forests' outputs are whole numbers, but for the out-of-bag error,
    a quotient of whole numbers that has no value without the forest."""
    if case["op"] not in ("surrogate_predict", "surrogate_grad"):
        return None
    P, mu, sd, lg = _network(seed)
    n = case["n_queries"] if case["op"] == "surrogate_predict" else case["batch"]
    X = _queries(n, seed + 7)
    p = torch.from_numpy(P).double().cuda().requires_grad_(case["op"] == "surrogate_grad")
    at = np.cumsum([0, HID * K_IN, HID, HID * HID, HID, HID, 1])
    w1, b1, w2, b2, w3, b3 = (p[a:b] for a, b in zip(at[:-1], at[1:]))

    def forward(X):
        gelu = torch.nn.functional.gelu
        h1 = gelu(_encode64(X, mu, sd, lg) @ w1.view(HID, K_IN).T + b1)
        return gelu(h1 @ w2.view(HID, HID).T + b2) @ w3 + b3

    if case["op"] == "surrogate_predict":
        return torch.cat([forward(X[:, i:i + 65536]) for i in range(0, n, 65536)])
    loss = 0.5 * (forward(X) - _targets(n, seed).double().cuda()).square().sum()
    (grad,) = torch.autograd.grad(loss / n, p)
    return dict(grad=grad, loss=loss.detach().reshape(1))

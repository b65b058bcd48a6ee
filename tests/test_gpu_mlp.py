"""The triage network's kernels (tcw_triage.cu) at batch sizes around their tiles
(64 rows, 32 rows of the output layer, eighths of the batch), against FP64
products of the same fp32 inputs.  Bounds: a chain of n fp32 FMAs errs by at
most (n + 2) u times the sum of its terms' magnitudes, u = 2^-24."""
import numpy as np
import pytest
import torch

import paper_2507_07816_gb300 as tcw
from oracle import triage as OT

pytestmark = pytest.mark.gpu
U = 2.0 ** -24


def close(got, ref, mag, n):
    assert got.shape == ref.shape
    assert np.all(np.abs(got - ref) <= (n + 2) * U * mag + 1e-37)


@pytest.mark.parametrize("n", [1, 7, 8, 31, 33, 63, 64, 65, 127, 129, 1030])
def test_forward_and_gradients(n):
    r = np.random.default_rng(900 + n)
    theta = (r.normal(size=OT.N_PARAMS) * 0.1).astype(np.float32)
    X = r.normal(size=(n, 128)).astype(np.float32)
    dy = r.normal(size=n).astype(np.float32)
    mlp = tcw.Mlp(theta)
    Xt = torch.as_tensor(X, device="cuda:0")
    H1t, H2t, yt = mlp.forward(Xt)
    g = OT.unpack(mlp.backward(Xt, H1t, H2t, torch.as_tensor(dy, device="cuda:0")).cpu().numpy().astype(np.float64))
    X, dy, H1, H2, y = (np.asarray(a, np.float64) for a in (X, dy, H1t.cpu(), H2t.cpu(), yt.cpu()))
    t = {k: v.astype(np.float64) for k, v in OT.unpack(theta).items()}
    W1, W2, w3 = (OT.bf16_round(t[k]).astype(np.float64) for k in ("W1", "W2", "w3"))
    w3 = w3.reshape(-1)
    close(H1, np.maximum(X @ W1 + t["b1"], 0), np.abs(X) @ np.abs(W1) + np.abs(t["b1"]), 128)
    close(H2, np.maximum(H1 @ W2 + t["b2"], 0), H1 @ np.abs(W2) + np.abs(t["b2"]), 256)
    close(y, H2 @ w3 + t["b3"][0], H2 @ np.abs(w3) + np.abs(t["b3"][0]), 256)
    dZ2 = dy[:, None] * w3 * (H2 > 0)
    dZ1, mZ1 = dZ2 @ W2.T * (H1 > 0), np.abs(dZ2) @ np.abs(W2).T * (H1 > 0)
    a = np.abs(dZ2)
    close(g["w3"].reshape(-1), H2.T @ dy, H2.T @ np.abs(dy), n)
    close(g["b3"].reshape(-1), dy.sum(keepdims=True), np.abs(dy).sum(keepdims=True), n)
    close(g["W2"], H1.T @ dZ2, H1.T @ a, n + 1)
    close(g["b2"].reshape(-1), dZ2.sum(0), a.sum(0), n + 1)
    close(g["W1"], X.T @ dZ1, np.abs(X).T @ mZ1, n + 258)
    close(g["b1"].reshape(-1), dZ1.sum(0), mZ1.sum(0), n + 258)


@pytest.mark.parametrize("n", [1, 31, 1025, 4096, 20000])
def test_loss(n):
    """Terms err by at most 10 u of their parts, their FP64 sum by one rounding."""
    r = np.random.default_rng(950 + n)
    y = (r.normal(size=n) * 4).astype(np.float32)
    label = (r.random(n) < 0.3).astype(np.float32)
    mlp = tcw.Mlp(seed=1)
    loss, dy = mlp.bce(torch.as_tensor(y, device="cuda:0"), torch.as_tensor(label, device="cuda:0"), 3.0)
    again, _ = mlp.bce(torch.as_tensor(y, device="cuda:0"), torch.as_tensor(label, device="cuda:0"), 3.0)
    ref, rdy = OT.bce_with_logits(y.astype(np.float64), label, pw=3.0)
    v = y.astype(np.float64)
    parts = np.mean(3.0 * label * (np.logaddexp(0, v) + np.abs(v)) + (1 - label) * np.logaddexp(0, v))
    assert abs(loss.item() - ref) <= 10 * U * parts + U * abs(ref)
    assert loss.item() == again.item()
    assert np.all(np.abs(dy.cpu().numpy() - rdy) <= 12 * U * 3.0 / n)

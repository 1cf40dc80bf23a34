"""Gradients of the preconditioner's network at the batch sizes where the
weight-gradient sums change form (one piece below 512 samples, then pieces of
at least 256, at most 32 of them) and at ragged tiles, against float64 with the
same bfloat16 weights.  Tolerance: sums of K float32 products with signs of
both kinds err by about sqrt(K) 2^-24 of their norm (K up to 8205 samples on
top of 256-long sums): 1e-5; a missing or doubled piece is off by 1e-2."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [1, 33, 511, 512, 530, 8205])
def test_gradients_match_float64(batch):
    import torch
    from paper_1408_5092_gb300 import _lib as L
    rng = np.random.default_rng(batch)
    shapes = {"W1": (256, 16), "b1": (256,), "W2": (256, 256), "b2": (256,), "W3": (2, 256), "b3": (2,)}
    p = {k: (rng.normal(size=s) * (0.05 if k[0] == "b" else np.sqrt(2.0 / s[1]))).astype(np.float32)
         for k, s in shapes.items()}
    x = rng.normal(size=(batch, 16)).astype(np.float32)
    t = rng.normal(size=(batch, 2)).astype(np.float32)
    net = L.mpspt_mlp_create()
    L.mpspt_mlp_set_params(net, p)
    loss, g = L.mpspt_mlp_gradient(net, x, t)
    L.mpspt_mlp_free(net)
    W = {k: torch.from_numpy(p[k]).bfloat16().double() for k in ("W1", "W2", "W3")}
    b = {k: torch.from_numpy(p[k]).double() for k in ("b1", "b2", "b3")}
    X, T = torch.from_numpy(x).double(), torch.from_numpy(t).double()
    h1 = torch.relu(X @ W["W1"].T + b["b1"])
    h2 = torch.relu(h1 @ W["W2"].T + b["b2"])
    y = h2 @ W["W3"].T + b["b3"]
    dy = (y - T) / batch
    d2 = (dy @ W["W3"]) * (h2 > 0)
    d1 = (d2 @ W["W2"]) * (h1 > 0)
    ref = {"W1": d1.T @ X, "b1": d1.sum(0), "W2": d2.T @ h1, "b2": d2.sum(0), "W3": dy.T @ h2, "b3": dy.sum(0)}
    assert abs(loss - float(0.5 * ((y - T) ** 2).sum() / batch)) <= 1e-5 * loss
    for k, r in ref.items():
        r = r.numpy()
        assert np.linalg.norm(g[k] - r) <= 1e-5 * np.linalg.norm(r), k

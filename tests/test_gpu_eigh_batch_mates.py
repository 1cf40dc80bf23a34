"""The mixed eigensolver where the largest matrix's rotation lists allow few
sweeps a launch (three at n = 1100): it and the small matrices beside it, to the
float64 bounds (1e-12 of the spectral radius; 4e-12 for n = 1100, whose rounding
grows with n as in the bound n eps)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_small_matrices_beside_a_large_one():
    import torch
    from paper_1408_5092_gb300 import _lib as L
    sizes = [30, 1100, 61, 240]
    mats = []
    for n in sizes:
        rng = np.random.default_rng(n)
        X = rng.normal(size=(n, n + 3))
        X[:, : n // 3] *= 1e-4
        mats.append(X @ X.T)
    A = torch.tensor(np.concatenate([m.ravel() for m in mats]), device="cuda", dtype=torch.float64)
    V, w = torch.zeros_like(A), torch.zeros(sum(sizes), device="cuda", dtype=torch.float64)
    L.mpspt_eigh_batched_ex(0, torch.cuda.current_stream().cuda_stream, sizes, A.data_ptr(), V.data_ptr(),
                            w.data_ptr(), 1)
    torch.cuda.synchronize()
    for n, m, v, e in zip(sizes, mats, torch.split(V, [n * n for n in sizes]), torch.split(w, sizes)):
        v, e = v.cpu().numpy().reshape(n, n), e.cpu().numpy()
        ref = np.linalg.eigvalsh(m)
        tol = 4e-12 if n == 1100 else 1e-12
        scale = np.abs(ref).max()
        assert np.max(np.abs(np.sort(e) - ref)) <= tol * scale, n
        assert np.max(np.abs(v.T @ v - np.eye(n))) <= tol, n
        assert np.max(np.abs(m @ v - v * e[None, :])) <= tol * scale, n

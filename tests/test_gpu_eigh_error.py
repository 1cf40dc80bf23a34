"""Errors of the eigensolvers' vectors against exact ones, over many small
matrices with eigenvalues spread over four decades (the spectra of a
truncation).  With C = V^T A V and G = V^T V in extended precision, the first
order error of vector j along i is (C_ij - G_ij w_j) / (w_j - w_i).  Bounds: the
geometric means over the same matrices that a float64 Jacobi solver with
rotations by divisions and square roots leaves (mixed: after a float32 start
and two Newton-Schulz steps, float64 sweeps on V^T A V)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _matrices(n, count):
    out = []
    for s in range(count):
        g = np.random.default_rng(1000 * n + s)
        lam = 10.0 ** (-4.0 * (np.arange(n) + 0.25 + 0.5 * g.random(n)) / n)
        Q = np.linalg.qr(g.normal(size=(n, n)))[0]
        M = (Q * (lam / lam.sum())) @ Q.T
        out.append(0.5 * (M + M.T))
    return np.array(out)


def _vector_error(A, V, w):
    A, V, w = (x.astype(np.longdouble) for x in (A, V, w))
    G, C = V.T @ V, V.T @ (A @ V)
    E = (C - G * w[None, :]) / (w[None, :] - w[:, None] + np.eye(len(w)))
    np.fill_diagonal(E, 0)
    return float(np.sqrt((E ** 2).sum(0)).max())


@pytest.mark.parametrize("entry,n,count,bound", [
    ("float64", 8, 1000, 1.301e-14), ("float64", 13, 1000, 5.271e-14), ("float64", 30, 500, 3.205e-13),
    ("mixed", 8, 1000, 6.099e-15), ("mixed", 13, 1000, 2.247e-14), ("mixed", 30, 500, 1.320e-13)])
def test_vector_errors(entry, n, count, bound):
    import torch
    from paper_1408_5092_gb300 import _lib as L
    A = _matrices(n, count)
    V, w = [], []
    for c in range(0, count, 250):
        a = torch.tensor(A[c:c + 250].ravel(), device="cuda")
        v, e = torch.empty_like(a), torch.empty(a.numel() // n, device="cuda", dtype=torch.float64)
        sizes = [n] * (a.numel() // (n * n))
        st = torch.cuda.current_stream().cuda_stream
        if entry == "mixed":
            L.mpspt_eigh_batched_ex(0, st, sizes, a.data_ptr(), v.data_ptr(), e.data_ptr(), 1)
        else:
            L.mpspt_eigh_batched(0, st, sizes, a.data_ptr(), v.data_ptr(), e.data_ptr())
        torch.cuda.synchronize()
        V.append(v.cpu().numpy().reshape(-1, n, n))
        w.append(e.cpu().numpy().reshape(-1, n))
    V, w = np.concatenate(V), np.concatenate(w)
    errs = [_vector_error(A[i], V[i], w[i]) for i in range(count)]
    assert np.exp(np.mean(np.log(errs))) <= bound

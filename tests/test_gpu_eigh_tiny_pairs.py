"""Couplings far below the float32 range of the matrix are rotated like any
other: 2 x 2 blocks of size 1e-40 to 1e-280 beside a block of size one, one size
per form of the float64 solver.  A block is one rotation in exact arithmetic, so
eigenvalues and vectors are within 16 units of rounding of their own size."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SCALES = [1.0, 1e-37, 1e-40, 1e-45, 1e-100, 1e-280]


@pytest.mark.parametrize("entry", ["mpspt_eigh_batched", "mpspt_eigh_batched_noalloc"])
@pytest.mark.parametrize("n", [12, 13, 40, 300, 601])
def test_tiny_blocks(entry, n):
    import torch
    from paper_1408_5092_gb300 import _lib as L
    rng = np.random.default_rng(n)
    ids = rng.permutation(n)[:2 * len(SCALES)].reshape(-1, 2)
    A, block = np.zeros((n, n)), np.array([[2.0, 0.5], [0.5, 1.0]])
    for ij, s in zip(ids, SCALES):
        A[np.ix_(ij, ij)] = s * block
    a = torch.tensor(A, device="cuda")
    V, w = torch.empty_like(a), torch.empty(n, device="cuda", dtype=torch.float64)
    getattr(L, entry)(0, torch.cuda.current_stream().cuda_stream, [n], a.data_ptr(), V.data_ptr(), w.data_ptr())
    torch.cuda.synchronize()
    V, w = V.cpu().numpy(), w.cpu().numpy()
    root = np.sqrt(0.5)          # eigenvalues 3/2 -+ root, vectors (root - 1/2, -1/2), (1/2, root - 1/2)
    want = np.array([[root - 0.5, 0.5], [-0.5, root - 0.5]]) / np.hypot(root - 0.5, 0.5)
    for ij, s in zip(ids, SCALES):
        lam, vec = w[ij], V[np.ix_(ij, ij)]
        o = np.argsort(lam)
        tol = 16 * 2.0 ** -53
        assert np.all(np.abs(lam[o] / s - np.array([1.5 - root, 1.5 + root])) <= tol * (1.5 + root))
        assert np.abs(np.abs(vec[:, o]) - np.abs(want)).max() <= tol

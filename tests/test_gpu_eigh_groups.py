"""Batches beyond one group of the mixed eigensolver (1 GiB of scratch: about
140 matrices of 236 x 236): every matrix to the float64 bounds, the second
group's small and large ones too, and twice in a row."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[236] * 170, [300, 20] * 6 + [236] * 160 + [301, 7]])
def test_more_than_one_group(sizes):
    import torch
    from paper_1408_5092_gb300 import _lib as L
    g = torch.Generator(device="cuda").manual_seed(5)
    mats = []
    for n in sizes:
        X = torch.randn(n, n + 3, device="cuda", dtype=torch.float64, generator=g)
        X[:, : n // 3] *= 1e-4
        mats.append(X @ X.T)
    A = torch.cat([m.reshape(-1) for m in mats])
    st = torch.cuda.current_stream().cuda_stream
    for _ in range(2):
        V, w = torch.zeros_like(A), torch.zeros(sum(sizes), device="cuda", dtype=torch.float64)
        L.mpspt_eigh_batched_ex(0, st, sizes, A.data_ptr(), V.data_ptr(), w.data_ptr(), 1)
        torch.cuda.synchronize()
        for n, m, v, e in zip(sizes, mats, torch.split(V, [n * n for n in sizes]), torch.split(w, sizes)):
            v = v.view(n, n)
            scale = float(e.abs().max())
            assert float((m @ v - v * e).abs().max()) <= 1e-12 * scale, n
            assert float((v.T @ v - torch.eye(n, device="cuda", dtype=torch.float64)).abs().max()) <= 1e-12, n
            assert abs(float(e.sum() - m.trace())) <= 1e-12 * n * scale, n

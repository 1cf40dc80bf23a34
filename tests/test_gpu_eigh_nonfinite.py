"""An infinity or a NaN in a matrix is never reported as converged: the calls
with a status return MPSPT_ERR_NOT_CONVERGED, the others leave NaN in that
matrix's w and V, and the other matrices of the batch are solved (float64
bounds as for the finite batches: 1e-12 of the spectral radius).  One size per
form of the solvers: one CTA, cluster, matrix beyond on-chip memory, mixed
sweeps in shared and in global memory."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _batch(n, bad, at):
    rng = np.random.default_rng(n)
    mats = []
    for m in (9, n, 33):
        X = rng.normal(size=(m, m + 2))
        mats.append(X @ X.T)
    mats[1][at] = mats[1][at[::-1]] = bad
    return mats


@pytest.mark.parametrize("at", [(1, 1), (0, 3)])
@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf")])
@pytest.mark.parametrize("n", [6, 40, 300, 600])
def test_non_finite_matrix(n, bad, at):
    import torch
    from paper_1408_5092_gb300 import _lib as L
    mats = _batch(n, bad, at)
    sizes = [m.shape[0] for m in mats]
    A = torch.tensor(np.concatenate([m.ravel() for m in mats]), device="cuda", dtype=torch.float64)
    st = torch.cuda.current_stream().cuda_stream
    for f32_start in (0, 1):
        V, w = torch.zeros_like(A), torch.zeros(sum(sizes), device="cuda", dtype=torch.float64)
        with pytest.raises(L.MpsptError) as e:
            L.mpspt_eigh_batched_ex(0, st, sizes, A.data_ptr(), V.data_ptr(), w.data_ptr(), f32_start)
        assert e.value.status == L.MPSPT_ERR_NOT_CONVERGED
    for call in (L.mpspt_eigh_batched, L.mpspt_eigh_batched_noalloc):
        V, w = torch.zeros_like(A), torch.zeros(sum(sizes), device="cuda", dtype=torch.float64)
        call(0, st, sizes, A.data_ptr(), V.data_ptr(), w.data_ptr())
        torch.cuda.synchronize()
        Vs = [v.cpu().numpy().reshape(m, m) for m, v in zip(sizes, torch.split(V, [m * m for m in sizes]))]
        ws = [v.cpu().numpy() for v in torch.split(w, sizes)]
        assert np.isnan(ws[1]).all() and np.isnan(Vs[1]).all()
        for q in (0, 2):
            scale = np.abs(np.linalg.eigvalsh(mats[q])).max()
            assert np.max(np.abs(mats[q] @ Vs[q] - Vs[q] * ws[q][None, :])) <= 1e-12 * scale
            assert np.max(np.abs(Vs[q].T @ Vs[q] - np.eye(sizes[q]))) <= 1e-12

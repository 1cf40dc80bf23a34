"""The float64 eigensolver on every kernel of its dispatch rule: batches of
equal matrices on both sides of each line (cluster, one CTA of 128, 256 and 512
threads), and a batch with sizes for all of them.  The kernels do the same
arithmetic per entry in the same order, so all copies of a matrix have the same
bits; float64 bounds as elsewhere (1e-12 of the spectral radius)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _matrix(n):
    rng = np.random.default_rng(n)
    X = rng.normal(size=(n, n + 3))
    X[:, : n // 3] *= 1e-4
    return X @ X.T


def _solve(sizes):
    import torch
    from paper_1408_5092_gb300 import _lib as L
    mats = {n: _matrix(n) for n in set(sizes)}
    A = torch.tensor(np.concatenate([mats[n].ravel() for n in sizes]), device="cuda", dtype=torch.float64)
    V, w = torch.zeros_like(A), torch.zeros(sum(sizes), device="cuda", dtype=torch.float64)
    L.mpspt_eigh_batched(0, torch.cuda.current_stream().cuda_stream, sizes, A.data_ptr(), V.data_ptr(), w.data_ptr())
    torch.cuda.synchronize()
    Vs = [v.cpu().numpy().reshape(n, n) for n, v in zip(sizes, torch.split(V, [n * n for n in sizes]))]
    ws = [v.cpu().numpy() for v in torch.split(w, sizes)]
    seen = {}
    for n, v, e in zip(sizes, Vs, ws):
        if n in seen:
            assert np.array_equal(v, seen[n][0]) and np.array_equal(e, seen[n][1]), n
            continue
        seen[n] = v, e
        ref = np.linalg.eigvalsh(mats[n])
        scale = np.abs(ref).max()
        assert np.max(np.abs(np.sort(e) - ref)) <= 1e-12 * scale, n
        assert np.max(np.abs(v.T @ v - np.eye(n))) <= 1e-12, n
        assert np.max(np.abs(mats[n] @ v - v * e[None, :])) <= 1e-12 * scale, n
    return seen


@pytest.mark.parametrize("n,batches", [(27, (1, 305)), (28, (38, 39, 305)), (33, (38, 39)), (64, (39, 305)),
                                       (65, (76, 77, 305)), (112, (76, 77)), (113, (113, 114)), (215, (114,)),
                                       (216, (2,))])
def test_equal_matrices(n, batches):
    first = None
    for b in batches:
        v, e = _solve([n] * b)[n]
        if first is None:
            first = v, e
        assert np.array_equal(v, first[0]) and np.array_equal(e, first[1]), b


def test_sizes_for_all_kernels_in_one_call():
    _solve([220, 60, 5] + [48] * 60 + [27, 28] * 20 + [1, 2])

"""The mixed eigensolver (float32 sweeps, float64 diagonal, float64 rounds)
where its branches change: matrix sizes at the edges of its thread counts (46,
92, 180) and of its shared-memory form (236), strongly graded and
rank-deficient spectra that need several rounds, repeated eigenvalues, and
scales far from one.  Bounds: a backward-stable float64 eigensolver is exact
to a small multiple of n eps of the spectral radius; 1e-12 covers n <= 300."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _graded(rng, n, decades):
    lam = 10.0 ** (-decades * (np.arange(n) + rng.uniform(0.2, 0.8, n)) / n)
    Q, _ = np.linalg.qr(rng.normal(size=(n, n)))
    A = (Q * lam) @ Q.T
    return 0.5 * (A + A.T)


def _solve(mats, f32_start):
    import torch
    from paper_1408_5092_gb300 import _lib as L
    sizes = [m.shape[0] for m in mats]
    A = torch.tensor(np.concatenate([m.ravel() for m in mats]), device="cuda", dtype=torch.float64)
    V = torch.zeros_like(A)
    w = torch.zeros(sum(sizes), device="cuda", dtype=torch.float64)
    L.mpspt_eigh_batched_ex(0, torch.cuda.current_stream().cuda_stream, sizes, A.data_ptr(), V.data_ptr(),
                            w.data_ptr(), f32_start)
    torch.cuda.synchronize()
    V, w = V.cpu().numpy(), w.cpu().numpy()
    o = ow = 0
    for n, m in zip(sizes, mats):
        v, e = V[o:o + n * n].reshape(n, n), w[ow:ow + n]
        scale = np.abs(m).max() * n if m.any() else 1.0
        ref = np.linalg.eigvalsh(m)
        scale = max(np.abs(ref).max(), 1e-300)
        assert np.max(np.abs(np.sort(e) - ref)) <= 1e-12 * scale, n
        assert np.max(np.abs(v.T @ v - np.eye(n))) <= 1e-12, n
        assert np.max(np.abs(m @ v - v * e[None, :])) <= 1e-12 * scale, n
        o += n * n
        ow += n


@pytest.mark.parametrize("f32_start", [0, 1])
@pytest.mark.parametrize("sizes", [[45, 46, 1, 2, 3], [47, 92, 91, 8], [93, 180, 5], [181, 236], [237, 12, 300]])
def test_sizes_at_the_edges_of_the_launch_rule(sizes, f32_start):
    rng = np.random.default_rng(sum(sizes))
    _solve([_graded(rng, n, 6) for n in sizes], f32_start)


@pytest.mark.parametrize("f32_start", [0, 1])
def test_spectra_that_need_several_rounds(f32_start):
    rng = np.random.default_rng(21)
    X = rng.normal(size=(64, 20))
    Q, _ = np.linalg.qr(rng.normal(size=(70, 70)))
    lam = np.repeat(rng.uniform(0, 1, 24), 3)[:70]
    mats = [_graded(rng, 80, 12), _graded(rng, 91, 16), X @ X.T, (Q * lam) @ Q.T, np.eye(16), np.zeros((9, 9)),
            np.diag(rng.normal(size=20)), np.ones((33, 33)), -_graded(rng, 30, 3)]
    mats += [_graded(rng, 40, 8) * 1e-30, _graded(rng, 41, 8) * 1e30]
    _solve(mats, f32_start)

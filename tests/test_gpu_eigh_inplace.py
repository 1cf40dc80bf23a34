"""Eigensolver calls whose outputs overlap their input give what separate
buffers give, bit for bit: V = A (all three entry points, one size per form of
the solver), and w inside A."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ENTRIES = [("mpspt_eigh_batched", ()), ("mpspt_eigh_batched_noalloc", ()), ("mpspt_eigh_batched_ex", (0,)),
           ("mpspt_eigh_batched_ex", (1,))]


@pytest.mark.parametrize("entry,extra", ENTRIES)
@pytest.mark.parametrize("sizes", [[13, 5], [40, 27], [400, 60], [600, 33]])
def test_outputs_over_the_input(entry, extra, sizes):
    import torch
    from paper_1408_5092_gb300 import _lib as L
    rng = np.random.default_rng(sum(sizes))
    mats = []
    for n in sizes:
        X = rng.normal(size=(n, n + 2))
        mats.append((X @ X.T).ravel())
    A = torch.tensor(np.concatenate(mats), device="cuda", dtype=torch.float64)
    st = torch.cuda.current_stream().cuda_stream
    V, w = torch.zeros_like(A), torch.zeros(sum(sizes), device="cuda", dtype=torch.float64)
    call = getattr(L, entry)
    call(0, st, sizes, A.data_ptr(), V.data_ptr(), w.data_ptr(), *extra)
    B, w2 = A.clone(), torch.zeros_like(w)
    call(0, st, sizes, B.data_ptr(), B.data_ptr(), w2.data_ptr(), *extra)
    C, V3 = A.clone(), torch.zeros_like(A)
    call(0, st, sizes, C.data_ptr(), V3.data_ptr(), C.data_ptr(), *extra)
    torch.cuda.synchronize()
    assert torch.equal(B, V) and torch.equal(w2, w)
    assert torch.equal(V3, V) and torch.equal(C[:w.numel()], w)

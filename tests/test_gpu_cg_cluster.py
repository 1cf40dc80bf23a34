"""Small local problems are solved by one launch on a thread-block cluster,
larger ones by launches per iteration.  Bond dimensions on both sides of the
line (single rows; every bond on the cluster; bonds of both kinds in one
sweep), direct and as graphs, against the oracle's sweep.  Tolerance: CG stops
at |r| <= 1e-10 |b| on either route, which moves the Hylleraas value by the
square of it; a near-degenerate truncation is the larger effect and the sweep
parity of this repository is 1e-8."""
import numpy as np
import pytest

import synthetic

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tiny():
    h, Lc, c = synthetic.config_integrals("tiny")
    ci, _ = synthetic.fci_reference(h, Lc, c["k_act"], c["n_elec"])
    return h, Lc, c, ci


def _run(L, tiny, M, **opts):
    h, Lc, c, ci = tiny
    o = L.mpspt_default_options()
    for k, v in opts.items():
        setattr(o, k, v)
    ctx = L.mpspt_create(o)
    L.mpspt_set_integrals(ctx, c["k_act"], h.shape[0] - c["k_act"], c["n_elec"], h, Lc)
    L.mpspt_set_reference_ci(ctx, ci)
    e2, _, rep = L.mpspt_minimize_hylleraas(ctx, "dyall", M, want_psi1=False)
    L.mpspt_destroy(ctx)
    return [rep.e2_per_sweep[s] for s in range(rep.n_sweeps)], rep


@pytest.mark.parametrize("M", [3, 9, 24, 40])
def test_solves_on_both_sides_of_the_line(tiny, M):
    import torch
    from oracle.mps import HylleraasSweep
    from oracle.operators import Problem
    from paper_1408_5092_gb300 import _lib as L
    h, Lc, c, ci = tiny
    base, rep = _run(L, tiny, M, max_sweeps=2, e_tol=1e-14)
    st = torch.cuda.Stream()
    graph, rg = _run(L, tiny, M, max_sweeps=2, e_tol=1e-14, stream=st.cuda_stream, cuda_graphs=1)
    assert graph == base and rg.cg_iters == rep.cg_iters
    p = Problem(h, Lc, c["k_act"], c["n_elec"], ci, h0="dyall")
    sw = HylleraasSweep(p, M, seed=1408)
    ref = [sw.sweep() for _ in range(2)]
    assert np.abs(np.array(base) - np.array(ref)).max() < 1e-8


@pytest.mark.parametrize("graphs", [0, 1])
def test_iteration_cap(tiny, graphs):
    import torch
    from paper_1408_5092_gb300 import _lib as L
    st = torch.cuda.Stream()
    with pytest.raises(L.MpsptError) as e:
        _run(L, tiny, 6, cg_max_iter=1, cg_tol=1e-15, stream=st.cuda_stream, cuda_graphs=graphs)
    assert e.value.status == L.MPSPT_ERR_NOT_CONVERGED

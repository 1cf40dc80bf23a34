"""Float64 grouped GEMM at the sizes where its tiling can go wrong: the Fig.
1C local operators at bond dimensions whose blocks are single rows, one row
or column past an 8 x 8 piece or a 16 x 16 / 32 x 32 tile, and K-lists that
are cut into pieces (medium chain), against the oracle.  Tolerance: a sum of
K products is exact to K eps times the sum of their absolute values; K < 1e3
here, so 1e-12 of the largest entry covers it."""
import numpy as np
import pytest

import synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [1, 8, 9, 17, 65])
def test_local_operators_at_tile_edges(M):
    from oracle.mps import HylleraasSweep, two_site_apply, two_site_mask
    from oracle.operators import Problem
    from paper_1408_5092_gb300 import _lib as L
    h, Lc, c = synthetic.config_integrals("tiny")
    ci, _ = synthetic.fci_reference(h, Lc, c["k_act"], c["n_elec"])
    p = Problem(h, Lc, c["k_act"], c["n_elec"], ci, h0="dyall")
    sw = HylleraasSweep(p, M, seed=13)
    ctx = L.mpspt_create()
    L.mpspt_set_integrals(ctx, c["k_act"], p.k - c["k_act"], c["n_elec"], h, Lc)
    L.mpspt_set_reference_ci(ctx, ci)
    psi = L.mpspt_mps_import(ctx, sw.psi1.A, sw.psi1.q)
    rng = np.random.default_rng(4)
    for i in (0, 2, 3, 7, p.k - 2):
        for s in range(i):
            sw._update_left(s)
        mask = two_site_mask(sw.psi1.q[i], sw.psi1.q[i + 2], sw.allowed.get(i + 1))
        x = rng.normal(size=mask.shape) * mask
        ref = two_site_apply(sw.LA[i], sw.WA.W[i], sw.WA.W[i + 1], sw.RA[i + 2], x, sw.WA.dims[i + 1]) * mask
        p0 = np.einsum("lsm,mtr->lstr", sw.psi0.A[i], sw.psi0.A[i + 1])
        rhs = two_site_apply(sw.LV[i], sw.WV.W[i], sw.WV.W[i + 1], sw.RV[i + 2], p0, sw.WV.dims[i + 1]) * mask
        got = L.mpspt_local_apply(ctx, "dyall", psi, i, L.MPSPT_LOCAL_SIGMA, x, x.shape)
        grhs = L.mpspt_local_apply(ctx, "dyall", psi, i, L.MPSPT_LOCAL_RHS, None, x.shape)
        assert np.abs(got - ref).max() <= 1e-12 * max(1.0, np.abs(ref).max()), i
        assert np.abs(grhs - rhs).max() <= 1e-12 * max(1.0, np.abs(rhs).max()), i
        sw.LA[1:] = [None] * (len(sw.LA) - 1)
        sw.LV[1:] = [None] * (len(sw.LV) - 1)
    L.mpspt_mps_free(psi)
    L.mpspt_destroy(ctx)

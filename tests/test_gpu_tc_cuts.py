"""Tensor-core local operator where its K-lists are cut: bond dimensions whose
K-lists end inside a stage of 64, fill one chunk, or go over several, on the
long chain (8 active + 24 virtual sites), against the float64 operator of the
same call.  Tolerance: the three-term bf16 split keeps 16 bits, 3 x 2^-17 =
2.3e-5 per product; sums of products of both signs leave up to a decade of the
largest entry, so 2e-4 of it."""
import numpy as np
import pytest

import synthetic

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def medium():
    h, Lc, c, ci = synthetic.config_reference("medium")
    return h, Lc, c, ci


def _apply(L, medium, prec, M, bonds):
    from oracle.mps import canonicalize_by_splits, random_mps, two_site_mask
    h, Lc, c, ci = medium
    k, N = h.shape[0], c["n_elec"]
    allowed = {c["k_act"]: {N - 1, N - 2}}
    psi1 = canonicalize_by_splits(random_mps(k, (N, 0), allowed, M, 5), allowed, 1e-10)
    o = L.mpspt_default_options()
    o.prec = L.PREC[prec]
    ctx = L.mpspt_create(o)
    L.mpspt_set_integrals(ctx, c["k_act"], k - c["k_act"], N, h, Lc)
    L.mpspt_set_reference_ci(ctx, ci)
    psi = L.mpspt_mps_import(ctx, psi1.A, psi1.q)
    rng = np.random.default_rng(2)
    out = []
    for i in bonds:
        mask = two_site_mask(psi1.q[i], psi1.q[i + 2], allowed.get(i + 1))
        x = rng.normal(size=mask.shape) * mask
        out.append(L.mpspt_local_apply(ctx, "dyall", psi, i, L.MPSPT_LOCAL_SIGMA, x, x.shape))
    L.mpspt_mps_free(psi)
    L.mpspt_destroy(ctx)
    return out


@pytest.mark.parametrize("M", [5, 31, 65])
def test_sigma_with_cut_k_lists(medium, M):
    from paper_1408_5092_gb300 import _lib as L
    bonds = (1, 4, 7, 8, 15, 29)
    for i, a, b in zip(bonds, _apply(L, medium, "fp64", M, bonds), _apply(L, medium, "mixed", M, bonds)):
        assert np.abs(a - b).max() <= 2e-4 * np.abs(a).max(), i

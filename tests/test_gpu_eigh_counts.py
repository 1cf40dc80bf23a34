"""The sweep counts of the verbose line are those of their phase: the polish
starts from V^T A V with an off-diagonal part of float32 rounding, so it takes a
fraction of the start's sweeps and at least one each round."""
import re

import pytest

import synthetic

pytestmark = pytest.mark.gpu


def test_polish_sweeps_do_not_include_the_start(capfd):
    from paper_1408_5092_gb300 import _lib as L
    h, Lc, c, ci = synthetic.config_reference("medium")
    o = L.mpspt_default_options()
    o.max_sweeps, o.verbose = 1, 3
    ctx = L.mpspt_create(o)
    L.mpspt_set_integrals(ctx, c["k_act"], h.shape[0] - c["k_act"], c["n_elec"], h, Lc)
    L.mpspt_set_reference_ci(ctx, ci)
    L.mpspt_minimize_hylleraas(ctx, "fock", 96, want_psi1=False)
    L.mpspt_destroy(ctx)
    m = re.findall(r"jacobi sweeps \(mean/max\): float32 ([\d.]+)/(\d+) polish ([\d.]+)/(\d+)", capfd.readouterr().err)
    assert m
    start, start_max, polish, polish_max = map(float, m[-1])
    assert 0.0 < polish < start and polish_max <= 8 * 60 and start_max <= 12

"""E3 of several first-order states on one context from several host threads at
once (each call waits for its own transfers; after a first call the operators
are there): the values of calls one after the other, bit for bit."""
import threading

import pytest

import synthetic

pytestmark = pytest.mark.gpu


def test_third_order_from_several_threads():
    from paper_1408_5092_gb300 import _lib as L
    h, Lc, c = synthetic.config_integrals("tiny")
    ci, _ = synthetic.fci_reference(h, Lc, c["k_act"], c["n_elec"])
    o = L.mpspt_default_options()
    o.max_sweeps = 2
    ctx = L.mpspt_create(o)
    L.mpspt_set_integrals(ctx, c["k_act"], h.shape[0] - c["k_act"], c["n_elec"], h, Lc)
    L.mpspt_set_reference_ci(ctx, ci)
    psis = [L.mpspt_minimize_hylleraas(ctx, "dyall", M)[1] for M in (6, 12, 20, 32)]
    want = [L.mpspt_third_order(ctx, "dyall", p) for p in psis]
    got = [[] for _ in psis]

    def work(i):
        for _ in range(10):
            got[i].append(L.mpspt_third_order(ctx, "dyall", psis[i]))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(psis))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for g, w in zip(got, want):
        assert g == [w] * 10
    for p in psis:
        L.mpspt_mps_free(p)
    L.mpspt_destroy(ctx)

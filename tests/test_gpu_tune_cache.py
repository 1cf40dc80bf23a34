"""The tuned-tile file: what it holds of the float64 kernel is one of that
kernel's two unit shapes (32 32 and 16 128)."""
import pytest

import synthetic

pytestmark = pytest.mark.gpu

F64 = 0   # first column of the file: the arithmetic


def _run(name, M, cache):
    from paper_1408_5092_gb300 import _lib as L
    h, Lc, c, ci = synthetic.config_reference(name)
    o = L.mpspt_default_options()
    o.max_sweeps, o.e_tol, o.autotune, o.autotune_cache = 1, 1e-14, 1, str(cache).encode()
    ctx = L.mpspt_create(o)
    L.mpspt_set_integrals(ctx, c["k_act"], h.shape[0] - c["k_act"], c["n_elec"], h, Lc)
    L.mpspt_set_reference_ci(ctx, ci)
    e2, _, _ = L.mpspt_minimize_hylleraas(ctx, "fock", M, want_psi1=False)
    L.mpspt_destroy(ctx)
    return e2, [tuple(map(int, line.split())) for line in cache.read_text().splitlines()]


def test_entries_of_other_tiles_are_timed_again(tmp_path):
    cache = tmp_path / "tiles.txt"
    e2, rows = _run("medium", 32, cache)
    f64 = [r for r in rows if r[0] == F64]
    assert f64 and all(r[6:] in ((32, 32), (16, 128)) for r in f64)
    for old in ((32, 64), (64, 64), (32, 32)):   # as files of the kernel's former tiles hold them
        cache.write_text("".join("%d %d %d %d %d %d %d %d\n" % ((r[:6] + old) if r[0] == F64 else r) for r in rows))
        again, new = _run("medium", 32, cache)
        assert {r[:6] for r in new} >= {r[:6] for r in rows}
        assert all(r[6:] in ((32, 32), (16, 128)) for r in new if r[0] == F64), old
        assert again == e2      # both unit shapes give the same bits


def test_small_float64_plans_are_not_timed(tmp_path):
    """Every float64 plan of the tiny system at M = 3 is below the step count under
    which the units are narrow whatever the tuner says."""
    cache = tmp_path / "tiles.txt"
    _, rows = _run("tiny", 3, cache)
    assert not [r for r in rows if r[0] == F64]

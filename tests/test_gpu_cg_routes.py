"""The two routes of a small local solve, told apart: sweeps of the tiny system
with the cluster launch available (every solve at M = 3, some at M = 40) and with
every such launch refused, direct and as graphs.  Both routes stop at |r| <= 1e-10
|b|, which moves the Hylleraas value by the square of it; the sweep parity of
this repository (a near-degenerate truncation is the larger effect) is 1e-8."""
import os
import subprocess

import numpy as np
import pytest

import synthetic

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def runs(tmp_path_factory):
    from paper_1408_5092_gb300 import _lib as L
    L.load()
    tmp = tmp_path_factory.mktemp("routes")
    h, Lc, c = synthetic.config_integrals("tiny")
    ci, _ = synthetic.fci_reference(h, Lc, c["k_act"], c["n_elec"])
    with open(tmp / "problem", "wb") as f:
        np.array([c["k_act"], h.shape[0] - c["k_act"], c["n_elec"], Lc.shape[0]], dtype=np.int64).tofile(f)
        for a in (h, Lc, ci):
            np.ascontiguousarray(a, dtype=np.float64).tofile(f)
    exe = tmp / "cg_routes"
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-I/usr/local/cuda/include",
                        os.path.join(ROOT, "tests", "cpp", "cg_routes.cpp"), L.LIB_PATH,
                        "-L/usr/local/cuda/lib64", "-lcudart", "-Wl,-rpath," + os.path.dirname(L.LIB_PATH),
                        "-Wl,-rpath,/usr/local/cuda/lib64", "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = subprocess.run([str(exe), str(tmp / "problem"), "3", "40"], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0, out.stdout + out.stderr
    res = {}
    for line in out.stdout.splitlines():
        v = line.split()
        res[tuple(map(int, v[:3]))] = dict(clusters=int(v[3]), launches=int(v[4]), iters=int(v[5]), calls=int(v[6]),
                                           flops=float(v[7]), e2=np.array(v[8:], dtype=float))
    assert len(res) == 8
    solves = 2 * 2 * (h.shape[0] - 1)   # sweeps, directions, bonds
    return res, solves


@pytest.mark.parametrize("M", [3, 40])
@pytest.mark.parametrize("graphs", [0, 1])
def test_refused_launches_take_the_other_route(runs, M, graphs):
    res, solves = runs
    on, off = res[M, graphs, 0], res[M, graphs, 1]
    assert on["clusters"] == solves if M == 3 else 0 < on["clusters"] < solves
    assert off["clusters"] == 0 and off["launches"] > on["launches"]
    assert np.abs(on["e2"] - off["e2"]).max() < 1e-8


@pytest.mark.parametrize("M", [3, 40])
@pytest.mark.parametrize("graphs", [0, 1])
def test_flops_of_one_launch_solves_are_not_counted(runs, M, graphs):
    """At M = 3 only the application that evaluates each solve is launched by
    itself; what refused runs launch by themselves is at least twice that."""
    res, _ = runs
    on, off = res[M, graphs, 0], res[M, graphs, 1]
    assert on["calls"] >= on["iters"] and 0 < on["flops"] < off["flops"]
    if M == 3:
        assert off["flops"] > 2 * on["flops"]

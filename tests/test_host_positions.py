"""Host check of the mixed Jacobi kernel's position addressing, compiled with
g++ from the GPU library's own header, for every even size up to 64."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_positions_follow_the_round_robin_order(tmp_path):
    exe = tmp_path / "positions_check"
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-I" + os.path.join(ROOT, "paper_1408_5092_gb300", "csrc"),
                        os.path.join(ROOT, "tests", "cpp", "positions_check.cpp"), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.split() == ["ok", "32"], out.stdout

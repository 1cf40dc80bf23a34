"""Host check of the staging ring's scopes, compiled with g++ from the library's
own header; no device is touched."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_a_ring_serves_one_scope_at_a_time(tmp_path):
    exe = tmp_path / "ring_check"
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-pthread", "-I/usr/local/cuda/include",
                        os.path.join(ROOT, "tests", "cpp", "ring_check.cpp"), "-L/usr/local/cuda/lib64", "-lcudart",
                        "-Wl,-rpath,/usr/local/cuda/lib64", "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.startswith("ok"), out.stdout + out.stderr

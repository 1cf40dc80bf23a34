"""Host check of the operators' element lists, linked against the built library;
no device is touched."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_lists_are_made_at_their_first_use(tmp_path):
    from paper_1408_5092_gb300 import _lib as L
    if not os.path.exists(L.LIB_PATH):
        from paper_1408_5092_gb300.build import build
        build()
    exe = tmp_path / "lists_check"
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-pthread", "-I/usr/local/cuda/include",
                        os.path.join(ROOT, "tests", "cpp", "lists_check.cpp"), L.LIB_PATH,
                        "-L/usr/local/cuda/lib64", "-lcudart", "-Wl,-rpath," + os.path.dirname(L.LIB_PATH),
                        "-Wl,-rpath,/usr/local/cuda/lib64", "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.startswith("ok"), out.stdout + out.stderr

"""Host check of the tensor-core kernel's float32 -> float64 conversion, compiled
with g++ from the GPU library's own header."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_every_float32_keeps_its_value(tmp_path):
    exe = tmp_path / "fconv_check"
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-I/usr/local/cuda/include",
                        "-I" + os.path.join(ROOT, "paper_1408_5092_gb300", "csrc"),
                        os.path.join(ROOT, "tests", "cpp", "fconv_check.cpp"), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.startswith("ok"), out.stdout

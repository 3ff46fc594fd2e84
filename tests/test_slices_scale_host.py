"""Host check of the scales and magnitudes behind the FP64 tensor-core products (tests/slices_scale_check.cpp)."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))


def test_scales_and_magnitudes_on_host(tmp_path):
    exe = str(tmp_path / "slices_scale_check")
    subprocess.run(["g++", "-O2", "-std=c++17", "-o", exe, os.path.join(HERE, "slices_scale_check.cpp")], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout

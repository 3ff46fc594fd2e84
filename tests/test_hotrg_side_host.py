"""Host check of the side a HOTRG step takes when a solver fails (tests/hotrg_side_check.cpp)."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))


def test_failed_side_is_not_taken(tmp_path):
    exe = str(tmp_path / "hotrg_side_check")
    subprocess.run(["g++", "-O2", "-std=c++17", "-o", exe, os.path.join(HERE, "hotrg_side_check.cpp")], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_the_step_reads_all_four_statuses():
    """The step takes its side through hotrg_side, from the statuses of both Gram matrices' blocks."""
    src = open(os.path.join(HERE, "..", "paper_2410_11596_gb300", "csrc", "hs_hotrg.cu")).read()
    assert "int hinfo[4]" in src and "hotrg_side(hinfo, " in src

"""The plane kernel's schedules with rows widened to whole memory sectors keep every row on them (planner, on the host)."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_2104_04731_b200", "csrc")


def test_widened_rows_stay_on_sectors(tmp_path):
    exe = str(tmp_path / "plane_sectors")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I", os.path.join(cuda, "include"), "-I", os.path.join(ROOT, "include"), "-I", CSRC,
                           os.path.join(HERE, "plane_sectors.cpp"), os.path.join(CSRC, "planner.cpp"), "-o", exe])
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr

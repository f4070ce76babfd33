"""The particle kernels' index arithmetic (divisions as multiplications, lattice sites) on the CPU, against the ordinary
divisions: every divisor up to 1024, the whole range of cell and particle indices and words beyond it."""
import os
import subprocess

from paper_1506_03737_gb300 import build


def test_index_arithmetic(tmp_path):
    here = os.path.dirname(os.path.abspath(__file__))
    exe = str(tmp_path / "host_index_check")
    subprocess.run([build._nvcc(), "-std=c++17", "-O2", "-o", exe, os.path.join(here, "host_index_check.cu")], check=True)
    res = subprocess.run([exe], capture_output=True, text=True)
    assert res.returncode == 0, res.stdout

"""A network whose bounded device-side wait gave up: no update from gradients that are not all there. The error word is set by
the test; nothing waits."""
import os
import subprocess

import pytest

from paper_1506_03737_gb300 import build

pytestmark = pytest.mark.gpu


def test_no_update_after_a_wait_that_gave_up(tmp_path):
    exe = str(tmp_path / "nn_timeout")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "gpu_nn_timeout_check.cu")
    subprocess.run([build._nvcc(), "-std=c++17", "-O1", *build.ARCH, "-I", build.CSRC, src, "-o", exe], check=True)
    res = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert res.returncode == 0, res.stdout

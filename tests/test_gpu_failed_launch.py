"""A launch that fails between others on the context's side streams."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu


def test_launches_before_a_failed_one_are_joined(tmp_path):
    from paper_1910_03936_gb300 import build
    here = os.path.dirname(os.path.abspath(__file__))
    exe = str(tmp_path / "failed_launch")
    subprocess.run([build._nvcc(), *build.ARCH, "-O2", "-std=c++17", "-I", build.INCLUDE, "-I", build.CSRC,
                    os.path.join(here, "native", "failed_launch.cu"),
                    os.path.join(build.CSRC, "pf_api.cu"), "-o", exe], check=True, timeout=300)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr

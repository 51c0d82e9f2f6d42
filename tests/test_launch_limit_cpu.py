"""The limit on the blocks of a fused launch, for the direct launches behind separable problems
(planning and tables only: a host program, no GPU)."""
import os
import shutil
import subprocess

import pytest

from paper_2103_09686_gb300 import _build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_gated_launches_count(tmp_path):
    nvcc = _build._nvcc()
    if shutil.which(nvcc) is None:
        pytest.skip("no nvcc")
    _build.build()
    objs = [os.path.join(_build.BUILD_DIR, os.path.splitext(s)[0] + ".o") for s in _build.SOURCES if s != "api.cu"]
    exe = str(tmp_path / "probe")
    subprocess.check_call([nvcc, *_build.ARCH, "-O0", "-std=c++17", "-I", _build.INCLUDE, "-I", _build.CSRC, "-o", exe,
                           os.path.join(ROOT, "tests", "launch_limit_probe.cu"), *objs])
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr

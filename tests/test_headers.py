"""Every kernel header compiles by itself (CPU)."""

import os
import subprocess

import pytest

from paper_2009_09500_gb300 import build


@pytest.mark.parametrize("header", sorted(f for f in os.listdir(build.CSRC) if f.endswith(".cuh")))
def test_header_stands_alone(header, tmp_path):
    src = tmp_path / "one.cu"
    src.write_text(f'#include "{header}"\n')
    cmd = [os.environ.get("NVCC", "nvcc"), *build.ARCH, "-std=c++17", "-I", build.CSRC, "-I", build.INCLUDE, "-cubin",
           "-Xcicc", "-O0", "-Xptxas", "-O0", "-o", str(tmp_path / "one.cubin"), str(src)]
    subprocess.run(cmd, check=True, capture_output=True, text=True)

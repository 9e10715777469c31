"""Kernels whose launch bounds leave no register to spare: the compiler says whether they spill."""
import os
import re
import subprocess

import pytest

from conftest import ROOT
from paper_2001_07710_b200.build import CSRC, NVCC_FLAGS

NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")


@pytest.mark.skipif(not os.path.exists(NVCC), reason="no nvcc")
def test_the_simplex_projection_does_not_spill(tmp_path):
    out = subprocess.run([NVCC] + NVCC_FLAGS + ["-Xptxas", "-v", "-c", os.path.join(CSRC, "admm.cu"), "-o", str(tmp_path / "admm.o")],
                         capture_output=True, text=True, check=True, cwd=ROOT)
    spills = re.findall(r"Compiling entry function '\w*k_simplex_project\w*'.*?(\d+) bytes spill stores, (\d+) bytes spill loads", out.stdout + out.stderr, re.S)
    assert len(spills) == 5 and all(s == ("0", "0") for s in spills), spills

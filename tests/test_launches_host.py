"""The chain of launches of a call: behind a launch that failed nothing is launched, and only what ran is counted."""
import os
import shutil
import subprocess

from conftest import ROOT

PROGRAM = r"""
#include "common.cuh"
#include <stdio.h>
int main() {
  pat::Launches l;
  int ran = 0;
  l.add_result([&] { ++ran; return cudaSuccess; });
  l.add_result([&] { ++ran; return cudaErrorInvalidValue; });
  l.add_result([&] { ++ran; return cudaSuccess; });
  printf("%d %d %d\n", ran, l.n, l.error == cudaErrorInvalidValue);
}
"""


def test_nothing_is_launched_behind_a_failed_launch(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    (tmp_path / "chain.cu").write_text(PROGRAM)
    exe = str(tmp_path / "chain")
    subprocess.check_call([nvcc, "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-I",
                           os.path.join(ROOT, "paper_2001_07710_b200", "csrc"), str(tmp_path / "chain.cu"), "-o", exe])
    assert subprocess.check_output([exe], text=True).split() == ["2", "1", "1"]

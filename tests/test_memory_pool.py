"""The memory that destroyed handles leave with the process (host logic): bounded, taken back where an allocation of the
library fails, and given back as a whole on request.  Checked through a small host-only program on a stand-in for the CUDA
runtime."""
import os
import shutil
import subprocess

from paper_2112_09335_b200 import build

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2112_09335_b200", "csrc")
CUDA_INCLUDE = os.path.join(os.path.dirname(os.path.dirname(shutil.which(build.nvcc_path()) or build.nvcc_path())), "include")


def compiled(tmp_path_factory, name):
    exe = str(tmp_path_factory.mktemp("harness") / name)
    subprocess.run(["g++", "-std=c++17", "-O1", "-fopenmp", "-I", CSRC, "-I", CUDA_INCLUDE, os.path.join(HERE, name + ".cpp"), "-o", exe],
                   check=True)
    return exe


def test_idle_memory_is_bounded_and_given_back(tmp_path_factory):
    out = subprocess.run([compiled(tmp_path_factory, "memory_pool_harness")], capture_output=True, text=True)
    assert out.stdout.strip() == "ok", out.stdout

"""The memory that destroyed handles leave with the process (host logic): bounded, taken back where an allocation of the
library fails, and given back as a whole on request.  Checked through a small host-only program on a stand-in for the CUDA
runtime.  And the threads its copies take."""
import os
import shutil
import subprocess

import pytest

from paper_2112_09335_b200 import build

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2112_09335_b200", "csrc")
CUDA_INCLUDE = os.path.join(os.path.dirname(os.path.dirname(shutil.which(build.nvcc_path()) or build.nvcc_path())), "include")


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("harness") / "memory_pool")
    subprocess.run(["g++", "-std=c++17", "-O1", "-fopenmp", "-I", CSRC, "-I", CUDA_INCLUDE, os.path.join(HERE, "memory_pool_harness.cpp"),
                    "-o", exe], check=True)
    return exe


def test_idle_memory_is_bounded_and_given_back(harness):
    out = subprocess.run([harness], capture_output=True, text=True)
    assert out.stdout.strip() == "ok", out.stdout


@pytest.mark.parametrize("allowed,bytes_,threads", [(1, 9 << 20, 1), (2, 9 << 20, 2), (16, 9 << 20, 8), (16, (1 << 20) - 1, 1)])
def test_copies_keep_to_the_callers_thread_count(harness, allowed, bytes_, threads):
    env = dict(os.environ, OMP_NUM_THREADS=str(allowed))
    out = subprocess.run([harness, str(bytes_)], capture_output=True, text=True, env=env, check=True)
    assert int(out.stdout) == threads

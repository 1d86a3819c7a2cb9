"""The memory kept between stores and a store's release (csrc/device_memory.cpp), on the CPU against a stand-in for the CUDA runtime."""
import os
import subprocess

import pytest

from paper_2411_04975_b200 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("device_memory") / "check")
    cuda = os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")))
    subprocess.check_call(["g++", "-O1", "-g", "-std=c++17", "-DSD_KEEP_SECONDS=0.3", "-I", build.CSRC, "-I", os.path.join(ROOT, "include"), "-isystem",
                           os.path.join(cuda, "include"), os.path.join(ROOT, "tests", "device_memory_check.cpp"),
                           os.path.join(build.CSRC, "device_memory.cpp"), "-o", out, "-pthread"])
    return out


@pytest.mark.parametrize("check", ["free_waits_for_the_owner", "kept_memory_goes_back_by_itself", "what_is_in_use_stays",
                                   "trim_gives_back_at_once", "many_threads", "a_forked_child_ends",
                                   "kept_memory_is_bounded", "no_host_memory_throws_nothing"])
def test_device_memory(program, check):
    p = subprocess.run([program, check], capture_output=True, text=True, timeout=60)
    assert p.returncode == 0, p.stderr

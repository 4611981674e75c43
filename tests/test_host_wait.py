"""Report slots (csrc/host_wait.h) on the CPU, against stand-ins for the three runtime calls they make."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("host_wait") / "host_wait_check")
    subprocess.check_call([os.environ.get("CXX", "g++"), "-O1", "-std=c++17", "-pthread",
                           "-I" + os.path.join(ROOT, "paper_2607_14541_b200", "csrc"), "-I" + os.path.join(CUDA, "include"),
                           "-o", exe, os.path.join(ROOT, "tests", "host_wait_check.cpp")])
    return exe


@pytest.mark.parametrize("case", ["cut_short", "answered", "no_memory"])
def test_a_slot_is_given_back_only_when_no_kernel_can_write_to_it(checker, case):
    """A call cut short by a failed launch waits for the kernels before it; an answered one does not wait again."""
    assert subprocess.run([checker, case], timeout=60).returncode == 0

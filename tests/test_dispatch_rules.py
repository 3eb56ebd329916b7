"""The choices between a CTA per state (robot) and the packed evaluation (csrc/rmp_internal.h), run
through a small C++ program built from the same header: lines that follow the device's SMs."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA_INC = "/usr/local/cuda/include"


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    if shutil.which("g++") is None or not os.path.isdir(CUDA_INC):
        pytest.skip("needs g++ and the CUDA headers")
    exe = str(tmp_path_factory.mktemp("rules") / "dispatch_check")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "include"),
                           "-I", os.path.join(ROOT, "paper_2301_08068_gb300", "csrc"),
                           "-I", CUDA_INC, os.path.join(ROOT, "tests", "dispatch_check.cpp"),
                           "-o", exe])

    def run(n, rays, sms):
        out = subprocess.run([exe], input="%d %d %d\n" % (n, rays, sms), capture_output=True,
                             text=True, check=True).stdout.split()
        return [int(v) for v in out]
    return run


@pytest.mark.parametrize("sms", [152, 76, 16])
def test_lines_follow_the_device(rules, sms):
    # batches: 1024 rays, 16 states an SM; rollouts: any number of few-ray robots
    assert rules(16 * sms, 1024, sms) == [1, 1] and rules(16 * sms + 1, 1024, sms) == [0, 1]
    assert rules(1, 1025, sms) == [0, 0] and rules(65536, 16, sms) == [0, 1]
    # robots of more rays: two an SM, at least a robot for every 64 rays
    assert rules(2 * sms, 64 * min(2 * sms, 64), sms)[1] == 1
    assert rules(2 * sms + 1, 1100, sms)[1] == 0
    assert rules(18, 1152, sms)[1] == (1 if 18 <= 2 * sms else 0) and rules(17, 1152, sms)[1] == 0
    assert rules(2 * sms, 4097, sms)[1] == 0

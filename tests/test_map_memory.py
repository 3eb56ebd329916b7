"""The rules for the memory of a map's box field (csrc/rmp_policy.h), run through a small C++
program built from the same header: a field never takes the last of the device's memory."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA_INC = "/usr/local/cuda/include"
GB = 1 << 30
TOTAL = 277 * GB


@pytest.fixture(scope="module")
def policy(tmp_path_factory):
    if shutil.which("g++") is None or not os.path.isdir(CUDA_INC):
        pytest.skip("needs g++ and the CUDA headers")
    exe = str(tmp_path_factory.mktemp("policy") / "map_memory_check")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "include"),
                           "-I", os.path.join(ROOT, "paper_2301_08068_gb300", "csrc"),
                           "-I", CUDA_INC, os.path.join(ROOT, "tests", "map_memory_check.cpp"),
                           "-o", exe])

    def run(lines):
        out = subprocess.run([exe], input="\n".join(lines) + "\n", capture_output=True,
                             text=True, check=True).stdout.split()
        return [int(v) for v in out]
    return run


@pytest.mark.parametrize("field,room,free,fits", [
    (32 << 20, 0, TOTAL, True),
    (32 * GB, 0, TOTAL, True),
    (32 * GB + 1, 64 * GB, TOTAL, False),           # past the largest field, whatever is free
    (GB, 0, GB + TOTAL // 16, True),                # a sixteenth stays free, and not a byte less
    (GB, 0, GB + TOTAL // 16 - 1, False),
    (32 << 20, 0, 0, False),
    (32 << 20, (32 << 20) - 1, 0, False),
    (32 << 20, 32 << 20, 0, True),                  # the pool holds it already
])
def test_box_field_leaves_memory(policy, field, room, free, fits):
    assert policy(["fits %d %d %d %d" % (field, room, free, TOTAL)]) == [int(fits)]


@pytest.mark.parametrize("live,largest,free", [
    (0, 0, 0), (500 << 20, 1, 1),
    (0, 90 << 20, 90 << 20), (3 * GB, 90 << 20, 90 << 20),   # one more map of the largest size
    (0, 5 * GB, 2 * GB), (7 * GB, 5 * GB, 2 * GB),  # the most
])
def test_pool_keeps_one_map(policy, live, largest, free):
    assert policy(["keep %d %d" % (live, largest)]) == [live + free + (64 << 20)]

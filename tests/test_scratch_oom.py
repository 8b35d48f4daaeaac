"""A request for implicit scratch that runs out of device memory part of the way, made again
when there is memory: the second either completes every array that the kernels are given or fails
again; none is left null behind a success. csrc/capi.cu on the host, with an allocator that
fails once at each allocation in turn (tests/scratch_oom)."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA_INC = "/usr/local/cuda/include"
ERR_OOM = 4


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    if not os.path.isdir(CUDA_INC):
        pytest.skip("CUDA headers not found")
    out = str(tmp_path_factory.mktemp("oom") / "scratch_oom")
    # the entry points go unused, and with them what they need of the kernels and the CUDA runtime
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-ffunction-sections", "-fdata-sections", "-Wl,--gc-sections",
                           "-I", CUDA_INC, os.path.join(ROOT, "tests", "scratch_oom", "scratch_oom.cpp"), "-o", out, "-ldl"])

    def run(*args):
        r = subprocess.run([out, *map(str, args)], check=True, capture_output=True, text=True)
        return [int(w) for w in r.stdout.split()]
    return run


@pytest.mark.parametrize("hexa", [0, 1], ids=["tet", "hex"])
@pytest.mark.parametrize("mixed,fd", [(0, 0), (1, 0), (0, 1)], ids=["fp64", "mixed", "matrix-free"])
def test_retry_after_out_of_memory(program, hexa, mixed, fd):
    first, second, missing, count = program(-1, hexa, mixed, fd)
    assert (first, second, missing) == (0, 0, 0) and count >= 11
    for at in range(count):
        first, second, missing, total = program(at, hexa, mixed, fd)
        assert first == ERR_OOM, at
        assert (second, missing) == (0, 0), (at, second, missing)
        assert total == count + 1, at           # nothing is allocated twice

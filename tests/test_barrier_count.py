"""The arrival count of the grid barrier in the one-launch GMRES (csrc/reduce.cuh): a barrier is
passed when all of its blocks have arrived and not before, also where the count wraps at 2^32.
Compiled for the host: no GPU."""
import ctypes as C
import subprocess

import pytest

from paper_2304_09485_gb300 import _native

SRC = r"""
#include "reduce.cuh"
// barrier `gen` of `blocks` blocks, `here` of which have arrived
extern "C" int passed(unsigned gen, unsigned blocks, unsigned here) {
  const unsigned want = gen * blocks, seen = (gen - 1) * blocks + here;
  return hgks::arrived(seen, want);
}
"""


@pytest.fixture(scope="module")
def passed(tmp_path_factory):
    d = tmp_path_factory.mktemp("barrier")
    src, so = str(d / "b.cu"), str(d / "libb.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.run([_native._nvcc(), *_native.ARCH, "-std=c++17", "-I", _native.CSRC, "-shared", "-Xcompiler", "-fPIC", "-o", so, src],
                   check=True, capture_output=True)
    lib = C.CDLL(so)
    lib.passed.argtypes = [C.c_uint] * 3
    return lib.passed


@pytest.mark.parametrize("blocks", [1, 2, 48, 152, 160])
def test_passed_by_all_and_only_by_all(passed, blocks):
    wrap = 2 ** 32 // blocks
    for gen in (1, 2, 1000, wrap // 2, wrap // 2 + 1, wrap - 1, wrap, wrap + 1, wrap + 2, 2 * wrap):
        g = gen % 2 ** 32
        assert all(not passed(g, blocks, here) for here in range(blocks))
        # the blocks that go on to the next barrier may have arrived there already
        assert all(passed(g, blocks, blocks + ahead) for ahead in range(blocks))

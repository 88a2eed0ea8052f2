"""The layout of what the tensor-core forms keep of a mesh (csrc/topology.hpp): the blocks' offsets, blocks of
M_i^-1, a table and gather blocks share one allocation, without overlap, aligned as the vector
loads and bulk copies that read them need, and no larger than their contents and the alignment."""
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_00619_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "topology.hpp"
int main(int argc, char** argv) {
  const bool digits = std::atoi(argv[1]);
  const size_t tail = std::atoi(argv[2]), gather = std::atoi(argv[3]);
  std::vector<int64_t> np(1, 0);
  for (int i = 4; i < argc; ++i) np.push_back(np.back() + std::atoi(argv[i]));
  const afe::BlockLayout L = digits ? afe::block_layout(np, afe::pd_words, tail, gather)
                                    : afe::block_layout(np, afe::minv_split_words, tail, gather);
  std::printf("%zu %zu %zu", L.tail, L.gather, L.bytes);
  for (int64_t p : L.ptr) std::printf(" %lld", (long long)p);
  return 0;
}
"""


@pytest.fixture(scope="module")
def layout(tmp_path_factory):
    cxx = os.environ.get("CXX", "g++")
    if shutil.which(cxx) is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("layout")
    src, exe = d / "layout.cpp", d / "layout"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-O1", "-std=c++17", "-I" + CSRC, str(src), "-o", str(exe)], check=True)

    def run(*args):
        out = subprocess.run([str(exe), *map(str, args)], check=True, capture_output=True, text=True).stdout
        return [int(x) for x in out.split()]
    return run


@pytest.mark.parametrize("digits", [0, 1])
@pytest.mark.parametrize("nodes", [[4], [15], [16, 17, 127, 128, 129, 640], [20] * 50, [1100, 5, 63, 64, 65]])
def test_parts_are_disjoint_aligned_and_tight(layout, digits, nodes):
    for tail, gather in ((0, 16), (2048, 1000), (512, 128)):
        t, g, size, *ptr = layout(digits, tail, gather, *nodes)
        n = np.array(nodes)
        tiles = (n + 15) // 16
        if digits:
            need = tiles ** 2 * 16 * 16 * 8 + 2 * n          # eight digits per entry, 16-bit exponents
        else:
            need = tiles * (tiles + 1) // 2 * 16 * 16 * 4 + n  # pairs of 16-bit values, 8-bit exponents
        have = np.diff(np.array(ptr)) * 4
        assert len(ptr) == len(nodes) + 1 and 8 * len(ptr) <= 4 * ptr[0] < 8 * len(ptr) + 128
        assert (have >= need).all() and (have < need + 128).all()
        assert all(4 * p % 128 == 0 for p in ptr)
        assert t == 4 * ptr[-1] and g == t + 4 * tail and g % 128 == 0
        assert size == g + gather

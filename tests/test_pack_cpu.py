"""The brick index and the breadth-first nodes of packed trees against the
uploaded cells, cell by cell (host code only)."""

import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "paper_2202_08614_gb300", "csrc")


@pytest.fixture(scope="module")
def pack_check(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("pack") / "pack_check")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I", SRC,
                    "-I", os.path.join(cuda, "include"), os.path.join(ROOT, "tests", "pack_check.cpp"),
                    os.path.join(SRC, "fpo_pack.cpp"), "-o", exe], check=True)
    return exe


# the smallest and the deepest grid of the index, and a tree coarser than its max_depth
@pytest.mark.parametrize("depth,max_depth", [(4, 4), (5, 5), (6, 12), (8, 9), (11, 11), (11, 12)])
def test_brick_index_matches_the_octree(pack_check, depth, max_depth):
    for seed in range(3):
        out = subprocess.run([pack_check, str(depth), str(max_depth), str(seed)], capture_output=True, text=True, check=True)
        assert int(out.stdout) == 0


# the index's size against the tree's: none past 256 bytes a leaf and 64 KB
@pytest.mark.parametrize("depth,leaves,index", [(3, 60, 0), (4, 1, 1), (8, 1, 1), (9, 1, 0), (9, 2047, 0), (9, 2048, 1),
                                                (10, 16383, 0), (10, 16384, 1), (11, 10, 0), (11, 131071, 0), (11, 131072, 1)])
def test_sparse_deep_trees_have_no_index(tmp_path, depth, leaves, index):
    src = tmp_path / "fits.cpp"
    src.write_text("""
#include <cstdio>
#include "fpo_internal.h"
using namespace fpo;
int main()
{
    const int D = %d;
    const uint32_t n = %du;
    std::vector<uint8_t> depth(n, (uint8_t)D);
    std::vector<uint32_t> xyz;
    for (uint32_t j = 0; j < n; ++j) xyz.insert(xyz.end(), {j %% (1u << D), j >> D, 0u});
    std::vector<float> coeffs(n);
    fpo_tree_desc t{};
    t.n_leaves = n;
    t.max_depth = D;
    t.leaf_depth = depth.data();
    t.leaf_xyz = xyz.data();
    t.coeffs = coeffs.data();
    t.aabb_size = 1.0;
    PackedTree p;
    std::string err;
    if (validate_and_pack(&t, 1, 1, &p, &err, false) != FPO_OK || p.perm.size() != n || p.nodes.empty()) return 3;
    std::printf("%%d", !p.top.empty());
    return 0;
}
""" % (depth, leaves))
    exe, cuda = str(tmp_path / "fits"), os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I", SRC, "-I", os.path.join(cuda, "include"),
                    str(src), os.path.join(SRC, "fpo_pack.cpp"), "-o", exe], check=True)
    assert subprocess.run([exe], capture_output=True, text=True, check=True).stdout == str(index)

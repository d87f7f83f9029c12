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

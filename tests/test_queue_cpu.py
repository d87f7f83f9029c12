"""The ray queue of the fused mode over camera frames of every shape, and which
walk a traversal takes (host code only; the frames of 2^26 tiles and more are a
few pixels wide or high)."""

import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "paper_2202_08614_gb300", "csrc")


@pytest.fixture(scope="module")
def queue_check(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("queue") / "queue_check")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I", SRC,
                    "-I", os.path.join(cuda, "include"), os.path.join(ROOT, "tests", "queue_check.cpp"), "-o", exe], check=True)
    return exe


@pytest.mark.parametrize("w,h", [(1, 1), (7, 9), (1921, 1081), (1, 2 ** 29 - 8), (1, 2 ** 29), (1, 2 ** 31 - 1),
                                 (2 ** 31 - 1, 1), (3, 700_000_001), (600_000_001, 3), (46340, 46340)])
def test_every_pixel_has_one_slot(queue_check, w, h):
    out = subprocess.run([queue_check, str(w), str(h)], capture_output=True, text=True, check=True)
    assert int(out.stdout) == 0


def test_the_compaction_schedule_walks_the_octree(tmp_path):
    # the pipeline's shared-memory estimate asks the rule that the launcher follows
    src, cuda = tmp_path / "walk.cpp", os.environ.get("CUDA_HOME", "/usr/local/cuda")
    src.write_text("""#include "fpo_internal.h"
using fpo::brick_walk;
static_assert(brick_walk(true, 32) && !brick_walk(true, 31) && !brick_walk(true, 1) && !brick_walk(false, 32), "");
""")
    subprocess.run(["g++", "-std=c++17", "-fsyntax-only", "-I", os.path.join(ROOT, "include"), "-I", SRC, "-I",
                    os.path.join(cuda, "include"), str(src)], check=True)
    api = open(os.path.join(SRC, "fpo_api.cu")).read()
    assert "traverse_smem_bytes(brick, trav_threads)" in api and api.count("traverse_smem_bytes(") == 1

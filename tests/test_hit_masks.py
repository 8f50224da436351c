"""A warp skips a splat only when none of its pixels would blend it (csrc/gsr_hit.h), also for long thin splats, whose
quadratic cancels. Plain C++, no GPU."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def hit_masks(tmp_path_factory):
    from paper_2507_15683_gb300 import build as B
    nvcc = shutil.which(B.NVCC) or "/usr/local/cuda/bin/nvcc"
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    exe = str(tmp_path_factory.mktemp("hit") / "hit_masks")
    cmd = ["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-I", B.CSRC, "-I", inc,
           os.path.join(HERE, "hit_masks.cpp"), "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return exe


@pytest.mark.parametrize("least,largest", [(0.55, 20), (20, 300), (300, 1000), (1000, 3000), (3000, 20000)])
def test_no_blending_block_is_left_out(hit_masks, least, largest):
    r = subprocess.run([hit_masks, str(least), str(largest), "300000"], capture_output=True, text=True, timeout=300)
    hits, missed, masked = map(int, r.stdout.split())
    assert hits > 100000 and missed == 0, (hits, missed)

"""bench.py's operation and byte counts against the code: the passes of a match that csrc/pmm.cu launches and the MMAs
of a tile, and the size of a Jacobian record."""
import os
import re

import bench

PMM = os.path.join(os.path.dirname(os.path.abspath(bench.__file__)), "paper_2507_15683_gb300", "csrc", "pmm.cu")


def test_match_tensor_flops():
    src = open(PMM).read()
    passes = len(re.findall(r"go\(k_pmm_(?:sums|argmax),", src))
    body = src[src.index("void mma_tile("):]
    mmas = body[:body.index("\n}")].count("mma_bf16(tmem,")  # each 128 x 128 x 16
    n = 128 * 50
    assert bench.pmm_tensor_flops(n) == passes * (n // 128) ** 2 * mmas * 2 * 128 * 128 * 16


def test_jacobian_record_size():
    src = open(os.path.join(os.path.dirname(PMM), "gsr_internal.h")).read()
    assert bench.JAC_FLOATS == int(re.search(r"kJacStride = (\d+)", src).group(1))

"""PnP at the edges of its compaction (blocks of 2,048 matches, words of 32), where the P3P samples find their matches by
rank in the validity bits: against the oracle, with the suite's own checks. Phase timing runs the same kernels in order on
one stream; its results must be the same bits.
"""
import numpy as np
import pytest
import torch

from oracle import pnp as OP
from tests.test_gpu_pnp import _check, _gpu, _synthetic, _words

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,alpha_lo", [(64, 0.5), (2047, 0.0), (2048, 0.2), (2049, 0.2), (4096, 0.0), (6177, 0.45)])
def test_samples_by_rank(gsr, n, alpha_lo):
    cam, _, T_r, depth, alpha, matches = _synthetic(100 + n, n=n, out_frac=0.2, alpha_lo=alpha_lo)
    if n > 4096:  # a whole block without depth: its ranks are empty
        alpha.reshape(-1)[matches[:2048, 2]] = 0.1
    words = _words(n, 40)
    o = OP.pnp_ransac(depth, alpha, cam, T_r, matches, words, refine_iters=5)  # the solver's default
    _check(_gpu(gsr, cam, T_r, depth, alpha, matches, words), o, cam, 2.0)


def test_in_order_and_beside_give_the_same_bits(gsr):
    cam, _, T_r, depth, alpha, matches = _synthetic(7)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    S = gsr.PnP(len(matches), 64)
    args = (cam, T_r, t(depth), t(alpha), t(matches), t(_words(7, 64).view(np.int32)))
    a = S.solve(*args)
    gsr.gs_pnp_set_timing(S.handle, True)
    b = S.solve(*args)
    S.close()
    np.testing.assert_array_equal(a["T"], b["T"])
    for k in ("inlier", "valid_index", "points", "hyp_counts"):
        assert torch.equal(a[k], b[k]), k
    found = a["hyp_counts"] >= 0
    assert torch.equal(a["hyp_poses"][found], b["hyp_poses"][found])

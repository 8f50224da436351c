"""PMM at the edges of its tiles (128 cells), row pairs (256 cells) and CTA ranges, on maps of independent random cells,
against the fp64 definition: log-sum-exps to 1e-5, and every row, column and coarse decision that is clear of ties.
"""
import numpy as np
import pytest
import torch

from oracle import pmm as OP

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hc,wc", [(1, 2), (1, 127), (2, 64), (3, 43), (5, 51), (16, 16), (1, 257), (16, 24), (5, 77),
                                   (47, 49), (53, 61)])
def test_coarse_decisions_by_cell_count(gsr, hc, wc):
    g = np.random.default_rng(hc * 1000 + wc)
    h, w = 8 * hc, 8 * wc
    cells = g.standard_normal((32, hc, wc)).astype(np.float32)
    fq = np.repeat(np.repeat(cells, 8, 1), 8, 2) + 0.1 * g.standard_normal((32, h, w)).astype(np.float32)
    fr = np.repeat(np.repeat(np.roll(cells, 1, 2), 8, 1), 8, 2) + 0.1 * g.standard_normal((32, h, w)).astype(np.float32)
    o = OP.coarse_pmm(fq, fr)
    m = gsr.Matcher(h, w)
    first = None
    for _ in range(2):  # the second match finds the first one's partials in the workspace
        r = {k: v.cpu().numpy() for k, v in m.match(torch.from_numpy(fq).cuda(), torch.from_numpy(fr).cuda()).items()}
        first = first or r
        for k in r:
            np.testing.assert_array_equal(r[k], first[k])
    m.close()
    np.testing.assert_allclose(r["lse_row"], o["lse_row"], rtol=1e-5)
    np.testing.assert_allclose(r["lse_col"], o["lse_col"], rtol=1e-5)
    rok, cok = ~o["row_flag"], ~o["col_flag"]
    np.testing.assert_array_equal(r["row_best"][rok], o["row_best"][rok])
    np.testing.assert_array_equal(r["col_best"][cok], o["col_best"][cok])
    clear = lambda s: {tuple(x) for x in s.tolist() if rok[x[0]] and cok[x[1]]}  # noqa: E731
    assert clear(r["coarse"]) == clear(o["matches"])

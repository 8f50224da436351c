"""Calls of every kind in turn on one scene (graphs captured on the second call of a size, tile counts left zero by the
scan, counters zeroed by the table's upload) give the bits of a fresh scene's first call, at tile counts around a scan
chunk (8,192) and after an overflow of the workspace.
"""
import numpy as np
import pytest
import torch

from paper_2507_15683_gb300 import synth

pytestmark = pytest.mark.gpu


def _scene(n=20000):
    return synth.aerial_scene(5, n, extent=(0.0, 200.0, 0.0, 200.0), n_clusters=20)


def _pose(k):
    return synth.look_pose((100.0 + 5 * k, 40.0, 60.0), 0.1 * k, 0.5)


def _same(a, b):
    for k in a:
        assert torch.equal(a[k], b[k]), k


@pytest.mark.parametrize("w,h", [(16, 16), (333, 251), (2048, 1024), (2064, 1024)])
def test_repeated_renders(gsr, w, h):
    cam = synth.camera(w, h, 0.7 * w)
    S = gsr.Scene(_scene())
    for k in (0, 1, 2, 0):  # plain, captured, replayed with another pose and other buffers
        F = gsr.Scene(_scene())
        want = F.render(cam, _pose(k))
        F.close()
        _same(S.render(cam, _pose(k)), want)
    S.close()


def test_calls_of_every_kind_in_turn(gsr):
    cams = [synth.camera(240, 136, 175.0), synth.camera(120, 68, 87.5)]
    S, F = gsr.Scene(_scene()), gsr.Scene(_scene())
    want = [F.render(c, _pose(0)) for c in cams]
    tgt = [(o["rgb"], o["depth"]) for o in want]
    grads = []
    for c, (a, b) in zip(cams, tgt):
        G = gsr.Scene(_scene())
        grads.append(G.render_pose_grad(c, _pose(1), a, b))
        G.close()
    for _ in range(3):
        for i, c in enumerate(cams):
            _same(S.render(c, _pose(0)), want[i])
            _same(S.render(c, _pose(0)), want[i])
            for _ in range(2):
                loss, grad = S.render_pose_grad(c, _pose(1), *tgt[i])
                assert loss == grads[i][0]
                np.testing.assert_array_equal(grad, grads[i][1])
            S.visibility(c, _pose(0))
        outs = [S.alloc_outputs(c) for c in cams]
        S.render_batch(cams, [_pose(0)] * 2, outs, graph=True)
        torch.cuda.synchronize()
        for o, r in zip(outs, want):
            _same(o, r)
    S.close()
    F.close()


def test_renders_after_a_workspace_overflow(gsr):
    n = 300000  # more records and pairs than the first guess for this scene and size
    sc = synth.tiny_scene(3, n=n)
    sc["scales"] = (sc["scales"] * 4).astype(np.float32)
    cam = synth.camera(512, 512, 500.0)
    S, F = gsr.Scene(sc), gsr.Scene(sc)
    small = synth.camera(64, 64, 500.0)
    for _ in range(2):
        S.render(small, np.eye(4))
    want = F.render(cam, np.eye(4))
    for _ in range(3):
        _same(S.render(cam, np.eye(4)), want)
    S.close()
    F.close()

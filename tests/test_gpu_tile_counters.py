"""The per-tile counters of the binning stand apart by a spacing that depends on the call's tile count, and each call
leaves them at zero for the next, whose spacing may be another; the projection stages 32 views at a time. The lists
must be the ones of a fresh scene's call on its own (bytes and whole numbers).
"""
import pytest
import torch

from paper_2507_15683_gb300 import synth

pytestmark = pytest.mark.gpu


def _scene(n=20000):
    return synth.aerial_scene(5, n, extent=(0.0, 200.0, 0.0, 200.0), n_clusters=20)


def _pose(k):
    return synth.look_pose((100.0 + 3 * k, 40.0, 60.0), 0.1 * k, 0.5)


def _same(a, b):
    for k in a:
        assert torch.equal(a[k], b[k]), k


def test_sizes_in_turn_across_the_spacings(gsr):
    # 4,096 / 4,160 / 8,192 / 8,256 / 16,384 / 16,512 tiles: both sides of each line, largest first and last
    sizes = [(2064, 2048), (1024, 1024), (1040, 1024), (2048, 1024), (16, 16), (2064, 1024), (2048, 2048), (2064, 2048)]
    S = gsr.Scene(_scene())
    for i, (w, h) in enumerate(sizes):
        cam = synth.camera(w, h, 0.7 * w)
        F = gsr.Scene(_scene())
        want = F.render(cam, _pose(i))
        pairs = F.status()[2]
        F.close()
        _same(S.render(cam, _pose(i)), want)
        assert S.status()[2] == pairs
    S.close()


@pytest.mark.parametrize("n_views", [31, 32, 33, 65])
def test_views_staged_in_groups(gsr, n_views):
    S = gsr.Scene(_scene())
    cams = [synth.camera(96 + 16 * (k % 3), 64, 80.0) for k in range(n_views)]
    poses = [_pose(k % 7) for k in range(n_views)]
    outs = [S.alloc_outputs(c) for c in cams]
    S.render_batch(cams, poses, outs)
    torch.cuda.synchronize()
    F = gsr.Scene(_scene())
    for c, T, o in zip(cams, poses, outs):
        _same(F.render(c, T), {k: v for k, v in o.items() if v is not None})
    F.close()
    S.close()

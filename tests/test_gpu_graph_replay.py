"""Synchronous calls that are replayed from a CUDA graph, in the states where the replay could differ from the plain
call."""
import numpy as np
import pytest
import torch

from paper_2507_15683_gb300 import synth

pytestmark = pytest.mark.gpu

CALLS = 40  # more plain calls than any size takes before it is captured


def _scene(n=20000):
    return synth.aerial_scene(5, n, extent=(0.0, 200.0, 0.0, 200.0), n_clusters=20)


def _pose(k):
    return synth.look_pose((100.0 + 5 * k, 40.0, 60.0), 0.1 * k, 0.5)


def test_sizes_and_kinds_in_turn(gsr):
    # ten sizes, renders and gradients: more keys than a scene keeps graphs, so that graphs are captured, replayed,
    # given up and captured again; every call has the bits of a scene that has captured nothing
    cams = [synth.camera(w, h, 0.7 * w) for w in (16, 100, 240, 333, 960) for h in (16, 251)]
    S = gsr.Scene(_scene())
    want, grads = [], []
    for c in cams:
        F = gsr.Scene(_scene())
        want.append([F.render(c, _pose(k)) for k in range(2)])
        grads.append(F.render_pose_grad(c, _pose(1), want[-1][0]["rgb"], want[-1][0]["depth"]))
        F.close()
    for runs in (2, 12, 2, 12):
        for c, w, (loss, grad) in zip(cams, want, grads):
            for k in range(runs):
                out = S.render(c, _pose(k & 1))
                for name, v in w[k & 1].items():
                    assert torch.equal(out[name], v), (c, k, name)
                got = S.render_pose_grad(c, _pose(1), w[0]["rgb"], w[0]["depth"])
                assert got[0] == loss
                np.testing.assert_array_equal(got[1], grad)
    S.close()


def test_empty_scene(gsr):
    S = gsr.Scene(synth.tiny_scene(0, n=0))
    cam = synth.camera(48, 33, 40.0)
    for k in range(CALLS):
        T = np.eye(4)
        T[0, 3] = 0.1 * k
        out = S.render(cam, T)
        assert float(out["alpha"].abs().max()) == 0.0 and float(out["rgb"].abs().max()) == 0.0
    loss, grad = S.render_pose_grad(cam, np.eye(4), out["rgb"], out["depth"])
    assert loss == 0.0 and not np.any(grad)
    S.close()


@pytest.mark.parametrize("what,n,scale,size", [("records", 200000, 1.0, 128), ("pairs", 4000, 12.0, 512)])
def test_replay_that_outgrows_the_workspace(gsr, what, n, scale, size):
    # captured and replayed at a pose that sees nothing, on the first guess of the workspace (65,536 records, eight
    # pairs each); then a replay needs more: the call is done again on a grown workspace, and the tile counters start
    # at zero afterwards
    sc = synth.tiny_scene(3, n=n)
    sc["scales"] = (sc["scales"] * scale).astype(np.float32)
    cam = synth.camera(size, size, float(size))
    away = np.diag([-1.0, 1.0, -1.0, 1.0])
    F = gsr.Scene(sc)
    want = F.render(cam, np.eye(4))
    tgt = (torch.full_like(want["rgb"], 0.5), torch.full_like(want["depth"], 5.0))
    grad = F.render_pose_grad(cam, np.eye(4), *tgt)
    F.close()

    def render(S):
        out = S.render(cam, np.eye(4))
        for k, v in want.items():
            assert torch.equal(out[k], v), k

    def gradient(S):
        loss, g = S.render_pose_grad(cam, np.eye(4), *tgt)
        assert loss == grad[0]
        np.testing.assert_array_equal(g, grad[1])

    for first, second in ((render, gradient), (gradient, render)):
        S = gsr.Scene(sc)
        for _ in range(CALLS):
            S.render(cam, away)
            S.render_pose_grad(cam, away, *tgt)
        assert S.status()[1] == 0
        first(S)
        _, records, pairs = S.status()
        assert records > 65536 if what == "records" else (records < 65536 and pairs > 8 * 65536)
        for _ in range(CALLS):
            second(S)
            first(S)
        S.close()

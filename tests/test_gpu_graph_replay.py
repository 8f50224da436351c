"""Synchronous calls that are replayed from a CUDA graph, in the states where the replay could differ from the plain
call."""
import numpy as np
import pytest
import torch

from paper_2507_15683_gb300 import synth

pytestmark = pytest.mark.gpu

CALLS = 40  # more plain calls than any size takes before it is captured


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

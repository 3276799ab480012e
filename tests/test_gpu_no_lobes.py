"""Gradients of arrays without entries."""
import numpy as np
import pytest

from paper_2410_11419_gb300 import synth

pytestmark = pytest.mark.gpu


def test_gradients_of_a_scene_without_lobes(gs3):
    """Arrays that hold a placeholder (no lobes) have the gradient 0, whatever their memory held."""
    import torch
    from paper_2410_11419_gb300 import render as R
    scene = synth.make_scene(5, 400, 0, "ball", mlp_width=32, mlp_hidden=2)
    cam, light = synth.camera_light_pair(5, 48, 48)
    ds = R.DeviceScene(scene)
    rd = R.Renderer(ds, 48, 48, 1 << 18)
    img = rd.render(cam, light)
    stale = [torch.full_like(ds.t[f], float("nan")) for f in ds.ARRAYS_DEV for _ in range(8)]
    del stale
    g = rd.backward(cam, light, torch.ones_like(img))
    for f in ("lobe_rot", "lobe_sigma", "lobe_amp"):
        assert np.all(g[f].cpu().numpy() == 0.0), f

"""The camera backward recovers a ray's transmittance by division, entry by entry:
an error that repeats from entry to entry grows with their number."""
import numpy as np
import pytest

from paper_2410_11419_gb300 import synth

pytestmark = pytest.mark.gpu


def test_equal_entries(gs3, oracle):
    """200 Gaussians at one place have one alpha at a pixel.  Correctly rounded, the
    forward's products and the backward's quotients are off by up to 2^-24 each,
    in either direction: 2^-24 / sqrt(3) sqrt(400) = 7e-7 (rms) at the front entry,
    and the entry's alpha, the refined shadow's sum and the shading add some 3e-7.
    A reciprocal's rounding (2^-24 / sqrt(3) rms over the pixels) that every
    entry repeats makes 200 times 3.4e-8."""
    import torch
    from oracle import torch_ref as TR
    from paper_2410_11419_gb300 import render as R
    n, side = 200, 16
    scene = synth.make_scene(3, n, 1, "ball", mlp_width=32, mlp_hidden=1)
    cam, light = synth.camera_light_pair(3, side, side)
    for f in ("mean_op", "scale", "rot"):
        getattr(scene, f)[:] = getattr(scene, f)[:1]
    scene.mean_op[:] = (0.0, 0.0, 0.0, -3.4)
    scene.scale[:, :3] = 0.5
    scene.albedo_d[:, :3] = 0.7
    ds = R.DeviceScene(scene)
    rd = R.Renderer(ds, side, side, 1 << 16)
    opts = R.opts_struct(ablate=7)
    rd.render(cam, light, opts)
    rel = []
    for y in range(3, 13, 2):
        for x in range(3, 13, 2):
            dimg = np.zeros((side, side, 3), np.float32)
            dimg[y, x] = 1.0
            got = rd.backward(cam, light, torch.from_numpy(dimg).cuda(), opts)["albedo_d"][0, 0].item()
            ref, _ = TR.grads_given_image_grad(scene, cam, light, dimg, oracle.Opts(ablate=7))
            want = ref["albedo_d"][0, 0]
            assert want > 0
            rel.append(got / want - 1)
    assert np.sqrt(np.mean(np.square(rel))) <= 2e-6

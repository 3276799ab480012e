"""Splats far wider than the image: rays that stopped, rays that have not reached
their last entry and rows outside the image take no part in them, on ragged
images, against the FP64 oracle and its gradients (the tolerances of the parity
and backward tests)."""
import numpy as np
import pytest

from paper_2410_11419_gb300 import synth
from tests.test_gpu_backward import _as_ref_layout, _compare, _gpu_grads
from tests.test_gpu_parity import check_float_stages, check_integer_stages, run_both

pytestmark = pytest.mark.gpu


def wide_scene(seed, n, scale, cam, light):
    """Opaque splats, and 24 wide ones behind them as the camera and as the light
    see them.  At a focal length of 70 pixels and a distance of 5 a scale of 1e5
    has a deviation of 1.4e6 pixels."""
    scene = synth.make_scene(seed, n, 2, "ball", mlp_width=32, mlp_hidden=2)
    g = np.random.default_rng(seed)
    scene.mean_op[24:, 3] = g.uniform(2.0, 4.2, n - 24)  # below the alpha clamp
    for i in range(24):
        eye = (cam.pos, light.pos)[i % 2]
        p = -eye / np.linalg.norm(eye) * (1.5 + 0.5 * g.random()) + 0.2 * g.standard_normal(3)
        scene.mean_op[i, :3] = p
        scene.mean_op[i, 3] = g.uniform(-2.0, 1.0)
        scene.scale[i, :3] = scale * g.uniform(0.7, 1.4, 3)
    return scene


@pytest.mark.parametrize("w,h", [(37, 51), (70, 41)])
@pytest.mark.parametrize("scale", [1e3, 1e5, 1e7, 4e8])
def test_wide_splats(gs3, oracle, w, h, scale):
    from oracle import torch_ref as TR
    cam, light = synth.camera_light_pair(w, w, h)
    scene = wide_scene(w, 600, scale, cam, light)
    g, fr = run_both(gs3, oracle, scene, cam, light)
    assert (fr["final_T"] < 1e-2).mean() > 0.05 and (fr["n_contrib"] < 600).any()
    check_integer_stages(g, fr)
    check_float_stages(g, fr)
    target = oracle.render(synth.perturbed(scene, 5), cam, light)["img"]
    dimg, _ = TR.image_grad_of_loss(fr["img"], target)
    ref, _ = TR.grads_given_image_grad(scene, cam, light, dimg)
    rep = _compare(_gpu_grads(scene, cam, light, dimg), _as_ref_layout(scene, ref))
    assert len(rep) == 14

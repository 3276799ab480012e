"""The camera backward by quarter tiles (small images) and by half tiles (912 tiles
and more on 152 SMs), with ragged right and lower edges, against the FP64 gradient
oracle (the tolerances of the backward test)."""
import numpy as np
import pytest

from paper_2410_11419_gb300 import synth
from tests.test_gpu_backward import _as_ref_layout, _compare, _gpu_grads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,w,h", [(300, 17, 5), (300, 37, 51), (400, 487, 470)])
def test_strips(gs3, oracle, n, w, h):
    from oracle import torch_ref as TR
    scene = synth.make_scene(n + w, n, 2, "ball", mlp_width=32, mlp_hidden=2)
    scene.mean_op[::3, 3] += np.float32(5.0)  # alpha at its clamp, rays that stop
    cam, light = synth.camera_light_pair(n, w, h)
    target = oracle.render(synth.perturbed(scene, 1), cam, light)["img"]
    dimg, _ = TR.image_grad_of_loss(oracle.render(scene, cam, light)["img"], target)
    ref, _ = TR.grads_given_image_grad(scene, cam, light, dimg)
    assert len(_compare(_gpu_grads(scene, cam, light, dimg), _as_ref_layout(scene, ref))) == 14

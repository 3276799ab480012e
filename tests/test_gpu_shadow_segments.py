"""The shadow splat and its backward where a light tile's list meets the ends
of its 256-entry segments and the rays' stops, on images with ragged tiles,
against the FP64 oracle and its gradients (the tolerances of the parity and
backward tests)."""
import numpy as np
import pytest

from paper_2410_11419_gb300 import synth
from tests.test_gpu_backward import _as_ref_layout, _compare, _gpu_grads
from tests.test_gpu_parity import check_float_stages, check_integer_stages, run_both

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,w,h,opaque", [(256, 16, 16, False), (257, 16, 16, False), (513, 16, 16, True),
                                          (2600, 40, 24, False), (2600, 40, 24, True)])
def test_segment_edges(gs3, oracle, n, w, h, opaque):
    from oracle import torch_ref as TR
    scene = synth.make_scene(n, n, 2, "ball", mlp_width=32, mlp_hidden=2)
    if opaque:  # alpha reaches its clamp, and rays stop inside segments
        scene.mean_op[::2, 3] += np.float32(7.0)
    cam, light = synth.camera_light_pair(n + 3, w, h)
    g, fr = run_both(gs3, oracle, scene, cam, light)
    check_integer_stages(g, fr)
    check_float_stages(g, fr)
    target = oracle.render(synth.perturbed(scene, 5), cam, light)["img"]
    dimg, _ = TR.image_grad_of_loss(fr["img"], target)
    ref, _ = TR.grads_given_image_grad(scene, cam, light, dimg)
    rep = _compare(_gpu_grads(scene, cam, light, dimg), _as_ref_layout(scene, ref))
    assert len(rep) == 14

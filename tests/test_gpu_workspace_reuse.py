"""What a workspace still holds after a backward."""
import pytest

from paper_2410_11419_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,res", [(1000, 64), (20000, 256)])
def test_shadow_reduce_after_backward(gs3, n, res):
    """The shadow partials of a frame outlive its backward: the reduction alone gives the same T."""
    import torch
    from paper_2410_11419_gb300 import _native as N, render as R
    scene = synth.make_scene(n, n, 2, "ball", mlp_width=32, mlp_hidden=2)
    cam, light = synth.camera_light_pair(n, res, res)
    rd = R.Renderer(R.DeviceScene(scene), res, res, 1 << 20)
    img = rd.render(cam, light).clone()
    T = rd.stage("T").clone()
    rd.backward(cam, light, torch.ones_like(img))
    rd.stage("T").zero_()
    out = rd.render_stages(cam, light, N.GS3_STAGE_SHADOW_REDUCE | N.GS3_STAGE_MLP | N.GS3_STAGE_CAMERA)
    torch.cuda.synchronize()
    assert torch.equal(rd.stage("T"), T) and torch.equal(out, img)

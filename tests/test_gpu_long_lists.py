"""The shadow splat and its backward over lists of tens of thousands of entries, whose
length chooses segments of 64, 128 and 256 entries (at most 1023 per tile, beyond
which the last takes the rest), against the FP64 oracle and its gradients (the
tolerances of the parity and backward tests)."""
import numpy as np
import pytest

from paper_2410_11419_gb300 import synth
from tests.test_gpu_backward import _as_ref_layout, _compare
from tests.test_gpu_parity import assert_close

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,length,rest", [(40000, 64, False), (80000, 128, False), (160000, 256, False),
                                           (290000, 256, True)])
def test_gradients(gs3, oracle, n, length, rest):
    import torch
    from oracle import torch_ref as TR
    from paper_2410_11419_gb300 import render as R
    # a tile of 3 x 3 pixels; splats of 0.03 pixels, so that an entry passes at few of them
    # and rays stay open through much of the list
    scene = synth.make_scene(n, n, 1, "ball", mlp_width=32, mlp_hidden=1)
    scene.scale[:, :3] *= np.float32(0.15)
    scene.mean_op[:, 3] -= np.float32(2.0 + np.log(n / 40000))
    cam, light = synth.camera_light_pair(n, 3, 3)
    far = np.linalg.norm(scene.mean_op[:, :3] - light.pos, axis=1) > 3.0  # rays stop among these
    scene.mean_op[far, 3] += np.float32(2.5)
    lowpass = float(np.float32(1e-3))
    fr = oracle.render(scene, cam, light, oracle.Opts(lowpass=lowpass))
    longest = int(np.diff(fr["light_tile_start"]).max())
    assert (longest > 1023 * length) if rest else (1023 * length // 2 < longest <= 1023 * length)
    ds = R.DeviceScene(scene)
    rd = R.Renderer(ds, 3, 3, 1 << 20)
    opts = R.opts_struct(lowpass=lowpass)
    img = rd.render(cam, light, opts)
    assert_close("shadow T", rd.stage("T").cpu().numpy().astype(np.float64), fr["T"], fr["T_bound"])
    assert_close("image", img.cpu().numpy().astype(np.float64), fr["img"], fr["img_bound"])
    stop = rd.stage("light_stop").cpu().numpy().view(np.uint32)
    assert fr["T_bound"].max() == 0 and ((stop > longest // 2) & (stop <= longest)).any()
    dimg = np.random.default_rng(n).standard_normal((3, 3, 3))
    ref, _ = TR.grads_given_image_grad(scene, cam, light, dimg, oracle.Opts(lowpass=lowpass))
    got = rd.backward(cam, light, torch.from_numpy(dimg.astype(np.float32)).cuda(), opts)
    rep = _compare({k: v.cpu().numpy() for k, v in got.items()}, _as_ref_layout(scene, ref))
    assert len(rep) == 14
    rd.check()
    ds.close()

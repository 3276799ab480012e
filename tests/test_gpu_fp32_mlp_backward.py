"""The networks' backward against the FP64 gradient oracle (the tolerances of
the backward test): every width and depth, row counts around the 128-row tiles,
and a scene whose rows pass in two batches."""
import numpy as np
import pytest

from paper_2410_11419_gb300 import synth
from tests.test_gpu_backward import _as_ref_layout, _compare, _gpu_grads

pytestmark = pytest.mark.gpu


def setup(oracle, width, hidden, act, n):
    from oracle import torch_ref as TR
    scene = synth.make_scene(width + hidden, n, 2, "ball", mlp_width=width, mlp_hidden=hidden, act=act)
    g = np.random.default_rng(n)
    for m in (scene.phi, scene.psi):
        m.biases = [g.uniform(-0.3, 0.3, b.shape).astype(np.float32) for b in m.biases]
    cam, light = synth.camera_light_pair(5, 48, 48)
    target = oracle.render(synth.perturbed(scene, 1), cam, light)["img"]
    dimg, _ = TR.image_grad_of_loss(oracle.render(scene, cam, light)["img"], target)
    return scene, cam, light, dimg, TR.grads_given_image_grad(scene, cam, light, dimg)[0]


@pytest.mark.parametrize("width,hidden,act,n", [
    (16, 1, synth.RELU, 129), (32, 1, synth.LEAKY_RELU, 127), (32, 4, synth.RELU, 300), (64, 1, synth.RELU, 128),
    (64, 3, synth.LEAKY_RELU, 129), (128, 1, synth.LEAKY_RELU, 257), (128, 4, synth.RELU, 500)])
def test_network_gradients(gs3, oracle, width, hidden, act, n):
    scene, cam, light, dimg, ref = setup(oracle, width, hidden, act, n)
    assert len(_compare(_gpu_grads(scene, cam, light, dimg), _as_ref_layout(scene, ref))) == 14


def test_two_batches_of_rows(gs3, oracle):
    """312,000 transparent Gaussians before the visible ones change no gradient:
    the visible rows lie in the second batch of 2432 tiles."""
    scene, cam, light, dimg, ref = setup(oracle, 64, 2, synth.RELU, 700)
    pad = synth.make_scene(3, 312000, 2, "ball", mlp_width=64, mlp_hidden=2)
    pad.mean_op[:, 3] = -100.0
    scene.n += pad.n
    for f in ("mean_op", "scale", "rot", "shade_rot", "albedo_d", "albedo_s"):
        setattr(scene, f, np.concatenate([getattr(pad, f), getattr(scene, f)], 0))
    for f in ("latent", "lobe_rot", "lobe_sigma", "lobe_amp"):
        setattr(scene, f, np.concatenate([getattr(pad, f), getattr(scene, f)], 1))
    gpu = _gpu_grads(scene, cam, light, dimg)
    nets = {k: ref[k] for k in ("phi_w", "phi_b", "psi_w", "psi_b")}
    assert len(_compare(gpu, nets)) == 4
    assert not gpu["mean_op"][:312000].any()
    assert len(_compare({"latent": gpu["latent"][0, 312000:]}, {"latent": ref["latent"][:, :4]})) == 1


@pytest.mark.parametrize("ablate", [0, 1, 8])
@pytest.mark.parametrize("shared", [False, True])
def test_every_gradient_is_overwritten(gs3, ablate, shared):
    """The caller's arrays may hold anything: the backward writes every element."""
    import torch
    from paper_2410_11419_gb300 import _native as N, render as R
    scene = synth.make_scene(6, 300, 3, "ball", mlp_width=32, mlp_hidden=2)
    if shared:
        scene.lobe_shared = True
        scene.lobe_rot, scene.lobe_sigma = scene.lobe_rot[:, 0].copy(), scene.lobe_sigma[:, 0].copy()
    cam, light = synth.camera_light_pair(2, 50, 34)
    ds, opts = R.DeviceScene(scene), R.opts_struct(ablate=ablate)
    rd = R.Renderer(ds, 50, 34, 1 << 18)
    dimg = torch.rand_like(rd.render(cam, light, opts))
    first = rd.backward(cam, light, dimg, opts)
    filled = {f: torch.full_like(ds.t[f], float("nan")) for f in N.GRAD_FIELDS}
    N.gs3_render_backward(ds.handle, R.camera_struct(cam), R.light_struct(light), opts, dimg, rd.ws, rd.cap, rd.bws,
                          filled, torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    rd.check()
    for f in N.GRAD_FIELDS:
        assert torch.isfinite(filled[f]).all(), f
        assert torch.allclose(filled[f], first[f], rtol=1e-4, atol=1e-6 * float(first[f].abs().max() + 1e-30)), f
    ds.close()

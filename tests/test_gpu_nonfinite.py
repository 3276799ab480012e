"""A Gaussian of infinite colour, or a pixel of infinite loss gradient, reaches only
the pixels and Gaussians that it contributes to: not the neighbours whose entries
and rays are evaluated together with it."""
import numpy as np
import pytest

from paper_2410_11419_gb300 import synth

pytestmark = pytest.mark.gpu

W, H = 37, 51


def scene_and_view(seed, wall=False):
    """300 Gaussians; wall: five opaque ones in front of the camera hide them all."""
    scene = synth.make_scene(seed, 300, 2, "ball", mlp_width=32, mlp_hidden=2, act=synth.LEAKY_RELU)
    cam, light = synth.camera_light_pair(seed, W, H)
    if wall:
        for i in range(5):
            scene.mean_op[i, :3] = cam.pos * np.float32((1.6 + 0.05 * i) / 3.0)
            scene.mean_op[i, 3] = 4.0
            scene.scale[i, :3] = 3.0
    return scene, cam, light


def render(scene, cam, light, env=False, mlp_dtype=0):
    import torch
    from paper_2410_11419_gb300 import render as R
    ds = R.DeviceScene(scene, mlp_dtype=mlp_dtype)
    rd = R.Renderer(ds, W, H, 1 << 18)
    img = rd.render_environment(cam, *synth.environment_lights(3, 3)) if env else rd.render(cam, light)
    torch.cuda.synchronize()
    return img.cpu().numpy()


@pytest.mark.parametrize("wall", [False, True])
@pytest.mark.parametrize("env", [False, True])
def test_infinite_colour_stays_in_its_pixels(gs3, env, wall):
    scene, cam, light = scene_and_view(4, wall)
    for g in range(250, 256):
        def with_albedo(x):
            scene.albedo_d[g, :3] = x
            return render(scene, cam, light, env)
        plain = with_albedo(0.5)
        takes = (with_albedo(1e30) != plain).any(axis=2)
        got = with_albedo(np.inf)
        scene.albedo_d[g, :3] = 0.5
        assert np.array_equal(got[~takes], plain[~takes])
        assert not np.isfinite(got[takes]).all(axis=1).any()
        assert not (wall and takes.any())


@pytest.mark.parametrize("mlp_dtype", [0, 1, 2])
@pytest.mark.parametrize("env", [False, True])
def test_not_a_number_from_a_network_stays_in_its_pixels(gs3, env, mlp_dtype):
    """Of the refined shadow and the residual of one Gaussian (its latent is not a number)."""
    scene, cam, light = scene_and_view(6)
    for g in range(100, 103):
        latent = scene.latent[0, g].copy()
        plain = render(scene, cam, light, env, mlp_dtype)
        scene.latent[0, g] = np.float32(3.0)
        other = render(scene, cam, light, env, mlp_dtype)
        scene.latent[0, g] = np.nan
        got = render(scene, cam, light, env, mlp_dtype)
        scene.latent[0, g] = latent
        takes = (other != plain).any(axis=2)
        assert np.array_equal(got[~takes], plain[~takes])


def grads(scene, cam, light, dimg, ablate=0):
    import torch
    from paper_2410_11419_gb300 import render as R
    ds = R.DeviceScene(scene)
    rd = R.Renderer(ds, W, H, 1 << 18)
    opts = R.opts_struct(ablate=ablate)
    rd.render(cam, light, opts)
    out = rd.backward(cam, light, torch.from_numpy(dimg).cuda(), opts)
    torch.cuda.synchronize()
    return {k: v.cpu().numpy() for k, v in out.items()}


def test_hidden_infinite_colours_leave_the_other_gradients(gs3):
    """Opaque Gaussians hide others, whose colours become infinite."""
    scene, cam, light = scene_and_view(4)
    scene.mean_op[:, 3] += np.float32(4.0)
    scene.scale[:, :3] *= np.float32(4.0)
    dimg = np.random.default_rng(0).standard_normal((H, W, 3)).astype(np.float32)
    want = grads(scene, cam, light, dimg)
    hidden = (want["albedo_d"] == 0).all(axis=1)
    assert hidden.sum() >= 10 and (~hidden).sum() >= 50
    scene.albedo_d[hidden, :3] = np.inf
    got = grads(scene, cam, light, dimg)
    for f in want:
        a, b = got[f], want[f]
        if f in ("lobe_rot", "lobe_sigma", "lobe_amp", "latent"):
            a, b = a[:, ~hidden], b[:, ~hidden]
        elif a.shape[0] == 300:
            a, b = a[~hidden], b[~hidden]
        # the order of the atomic sums differs between runs
        assert np.isfinite(a).all() and np.linalg.norm(a - b) <= 1e-5 * np.linalg.norm(b), f


# no shadow splat and networks: a Gaussian meets a pixel through the camera alone;
# no networks: through the shadow splat as well
@pytest.mark.parametrize("ablate", [7, 6])
def test_infinite_pixel_gradient_stays_with_its_gaussians(gs3, ablate):
    scene, cam, light = scene_and_view(8)
    scene.mean_op[:, 3] += np.float32(1.0)
    for y, x in ((20, 17), (33, 9)):
        dimg = np.zeros((H, W, 3), np.float32)
        dimg[y, x] = (0.3, 1.0, 0.7)
        one = grads(scene, cam, light, dimg, ablate)
        dimg = np.random.default_rng(1).standard_normal((H, W, 3)).astype(np.float32)
        dimg[y, x] = np.inf
        got = grads(scene, cam, light, dimg, ablate)
        for f in ("mean_op", "scale", "albedo_d"):
            meets = (one[f] != 0).any(axis=1)
            assert np.isfinite(got[f][~meets]).all(), f
            assert meets.sum() < 290 and not np.isfinite(got[f][meets]).all()


def test_infinite_colour_in_a_batch(gs3):
    """Frames of a batch keep their own form: each equals its frame rendered alone, bit for bit."""
    import torch
    from paper_2410_11419_gb300 import _native as N, render as R
    scene, cam, light = scene_and_view(4)
    scenes = [R.DeviceScene(scene)]
    scene.albedo_d[250, :3] = np.inf
    scenes.append(R.DeviceScene(scene))
    server = R.Server(hbm_budget=1 << 30, max_inflight=1, max_batch=4)
    ids = [server.add_scene(x) for x in scenes]
    out = [torch.zeros((H, W, 3), device="cuda") for _ in range(8)]
    torch.cuda.synchronize()
    tickets = [server.submit(ids[i % 2], cam, light, x) for i, x in enumerate(out)]
    assert all(server.wait(t)[0] == N.GS3_OK for t in tickets)
    server.close()
    for i, x in enumerate(out):
        alone = R.Renderer(scenes[i % 2], W, H, 1 << 18).render(cam, light)
        assert torch.equal(x.view(torch.int32), alone.view(torch.int32))
        assert bool(torch.isfinite(x).all()) == (i % 2 == 0)

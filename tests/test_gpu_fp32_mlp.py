"""The FP32 networks' kernels against float64 at the same inputs: every width
and depth, row counts around the 128-row tiles and more tiles than SMs."""
import math

import numpy as np
import pytest

from paper_2410_11419_gb300 import synth

pytestmark = pytest.mark.gpu


def pe(v):
    return np.concatenate([v] + [f(2.0 ** q * math.pi * v) for q in range(4) for f in (np.sin, np.cos)], 1)


def network(m, x):
    for i, (w, b) in enumerate(zip(m.weights, m.biases)):
        x = x @ w.astype(np.float64).T + b.astype(np.float64)
        if i + 1 < len(m.weights):
            x = np.where(x > 0, x, 0.01 * x if m.act == synth.LEAKY_RELU else 0.0)
    return 1 / (1 + np.exp(-x))


@pytest.mark.parametrize("width,hidden,act,n", [
    (16, 2, synth.RELU, 300), (32, 1, synth.LEAKY_RELU, 1), (32, 3, synth.RELU, 127), (64, 2, synth.RELU, 128),
    (64, 4, synth.LEAKY_RELU, 129), (128, 1, synth.RELU, 1000), (128, 3, synth.LEAKY_RELU, 257),
    (128, 4, synth.RELU, 20000)])
def test_fp32_networks(gs3, width, hidden, act, n):
    import torch
    from paper_2410_11419_gb300 import render as R
    scene = synth.make_scene(width + hidden, n, 1, "ball", mlp_width=width, mlp_hidden=hidden, act=act)
    g = np.random.default_rng(n)
    for m in (scene.phi, scene.psi):
        m.biases = [g.uniform(-0.3, 0.3, b.shape).astype(np.float32) for b in m.biases]
    cam, light = synth.camera_light_pair(7, 64, 64)
    ds = R.DeviceScene(scene)
    rd = R.Renderer(ds, 64, 64, 1 << 20)
    rd.render(cam, light)
    torch.cuda.synchronize()
    rd.check()
    mu = scene.mean_op[:, :3].astype(np.float64)
    rest = np.concatenate([pe(mu), scene.latent[0], scene.latent[1][:, :2]], 1)
    unit = lambda d: d / np.linalg.norm(d, axis=1, keepdims=True)
    T = rd.stage("T").cpu().numpy().astype(np.float64)
    phi = network(scene.phi, np.concatenate([T[:, None], pe(unit(light.pos.astype(np.float64) - mu)), rest], 1))
    psi = network(scene.psi, np.concatenate([pe(unit(cam.pos.astype(np.float64) - mu)), rest], 1))
    # the direction's rounding (2^-23) grows by 8 pi in the highest band, and
    # each layer rounds sums of up to 128 products of order 1: about 1e-6 on the
    # pre-activations of a few, times the sigmoid's slope of at most 1/4
    tol = 2e-6
    assert np.abs(rd.stage("Tp").cpu().numpy() - phi[:, 0]).max() <= tol
    assert np.abs(rd.stage("res")[:, :3].cpu().numpy() - psi).max() <= tol
    ds.close()

"""Frames of networks of different shapes from several host threads."""
import threading

import pytest

from paper_2410_11419_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mlp_dtype", [0, 1, 2])
def test_networks_of_different_shapes(gs3, mlp_dtype):
    import torch
    from paper_2410_11419_gb300 import render as R
    errors = []

    def frames(width, hidden):
        try:
            scene = synth.make_scene(width, 200, 1, "ball", mlp_width=width, mlp_hidden=hidden)
            cam, light = synth.camera_light_pair(width, 32, 32)
            ds = R.DeviceScene(scene, mlp_dtype=mlp_dtype)
            rd = R.Renderer(ds, 32, 32, 1 << 14)
            stream = torch.cuda.Stream()
            stream.wait_stream(torch.cuda.current_stream())
            rd.render(cam, light, stream=stream)
            stream.synchronize()
            want = rd.image.cpu()
            for i in range(600):
                rd.render(cam, light, stream=stream)
                if i % 100 == 99:
                    stream.synchronize()
                    assert torch.equal(rd.image.cpu(), want)
            stream.synchronize()
            rd.header(stream)
        except Exception as e:  # reported by the test's thread
            errors.append(repr(e))

    threads = [threading.Thread(target=frames, args=a) for a in ((128, 4), (32, 1), (64, 3), (32, 2))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors

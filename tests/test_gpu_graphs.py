"""Frames and training views under stream capture."""
import pytest

from paper_2410_11419_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1000, 6000])
@pytest.mark.parametrize("mlp_dtype", [0, 1])
def test_captured_frame_and_backward(gs3, n, mlp_dtype):
    """A graph of a frame, its backward and a moved view under the same light replays what the
    calls give: both depth sorts (4096 keys), launches behind event waits, forks and joins."""
    import torch
    from paper_2410_11419_gb300 import _native as N, render as R
    stages = N.GS3_STAGE_PREP | N.GS3_STAGE_CAMERA_BIN | N.GS3_STAGE_MLP | N.GS3_STAGE_CAMERA
    scene = synth.make_scene(n, n, 2, "ball", mlp_width=32, mlp_hidden=2)
    cam, light = synth.camera_light_pair(n, 96, 80)
    cam2, _ = synth.camera_light_pair(n + 1, 96, 80)
    rd = R.Renderer(R.DeviceScene(scene, mlp_dtype=mlp_dtype), 96, 80, 1 << 18)
    dimg = torch.rand((80, 96, 3), device="cuda", generator=torch.Generator("cuda").manual_seed(n))
    out = [torch.empty((80, 96, 3), device="cuda") for _ in range(2)]

    def calls():
        rd.render(cam, light, out=out[0])
        g = rd.backward(cam, light, dimg)
        rd.render_stages(cam2, light, stages, out=out[1])
        return g

    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        want = {k: v.clone() for k, v in calls().items()}
        images = [x.clone() for x in out]
    stream.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        got = calls()
    for x in out:
        x.zero_()
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    rd.check()
    for a, b in zip(out, images):
        assert torch.equal(a, b)
    for f in want:  # the order of the atomic sums differs between runs
        assert (got[f] - want[f]).norm() <= 1e-5 * want[f].norm(), f

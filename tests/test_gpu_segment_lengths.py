"""The shadow segments' lengths of 64, 128 and 256 entries, which a frame's pair
count chooses (the smallest with at most 8192 segments' worth of pairs), against
the FP64 oracle with the tolerances of the parity test."""
import numpy as np
import pytest

from paper_2410_11419_gb300 import synth
from tests.test_gpu_parity import check_float_stages, check_integer_stages, run_both

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,length", [(6000, 64), (12000, 128), (24000, 256)])
def test_segment_lengths(gs3, oracle, n, length):
    scene = synth.make_scene(n, n, 1, "ball", mlp_width=32, mlp_hidden=1)
    scene.scale[:, :3] *= np.float32(6.0)
    scene.mean_op[:, 3] -= np.float32(3.0)  # faint: rays stay open through long lists
    cam, light = synth.camera_light_pair(n, 256, 240)
    g, fr = run_both(gs3, oracle, scene, cam, light, cap=1 << 21)
    pairs = g["hdr"].pairs_light
    assert pairs // length <= 8192 < pairs // (length // 2)
    check_integer_stages(g, fr)
    check_float_stages(g, fr)

"""Batches of a Gaussian count that is no multiple of four: a camera's records
start at a multiple of n inside the group's arrays, so its depth order is not
16-byte aligned."""
import numpy as np
import pytest

from paper_2605_04844_gb300 import synth

from gpu_util import to_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 4097, 20_001, 20_003])
def test_batch_of_odd_count_matches_frames(n):
    import torch
    from paper_2605_04844_gb300 import rasterizer as R
    scene = synth.scene_ball(n, 71, radius=3.0, deg=1)
    cams = [synth.pinhole(W, H, viewmat=synth.look_at((6.0 * np.sin(k), 0.5, -6.0 * np.cos(k)), (0.0, 0.0, 0.0)))
            for k, (W, H) in enumerate([(96, 64), (130, 70), (200, 120)])]
    sd = to_device(scene)
    b = R.calibrated_batch(sd, cams, group=3)
    b.render(R.scene_struct(sd), R.camera_array(cams), "quadbox", bg=(0.1, 0.2, 0.3))
    torch.cuda.synchronize()
    b.check()
    for k, c in enumerate(cams):
        img, _ = R.forward(sd, c, "quadbox", bg=(0.1, 0.2, 0.3))
        np.testing.assert_array_equal(b.image(k).cpu().numpy(), img.cpu().numpy())

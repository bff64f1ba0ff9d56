"""The batch's workspace, where the binning of a group shares its memory with
the pixels' state and the sums of the backward, and the cell ids lie in the
cameras' slots: images and gradients equal those of frames, call after call on
one batch, with cell ids of one and of two passes, with as many sets as cameras
and fewer, with groups of several cameras and of one, on both sides of the limit
between the two depth sorts, and for Gaussian counts that align nothing."""
import numpy as np
import pytest

from paper_2605_04844_gb300 import synth

from gpu_util import to_device

pytestmark = pytest.mark.gpu

KEYS = ("means", "scales", "quats", "opacities", "sh")
SMALL = [(130, 70), (64, 64), (200, 120), (50, 90), (96, 64), (33, 17), (80, 60), (150, 40), (48, 48), (120, 100)]
WIDE = [(2560, 1440), (320, 200), (2570, 1300)]  # the largest: ids of two passes at 8 bits


def cameras(sizes, turn):
    return [synth.pinhole(W, H, viewmat=synth.look_at((6.0 * np.sin(k + turn), 0.7, -6.0 * np.cos(k + turn)),
                                                      (0.0, 0.0, 0.0))) for k, (W, H) in enumerate(sizes)]


def grads_of(sd):
    import torch
    from paper_2605_04844_gb300 import _native as N
    g = {k: torch.zeros_like(sd[k]) for k in KEYS}
    gs = N.QbSceneGrads()
    for k in KEYS:
        setattr(gs, k, g[k].data_ptr())
    return g, gs


@pytest.mark.parametrize("n,sizes,group,tune", [
    (5001, SMALL, 10, None),                          # more cameras than sets
    (40_003, SMALL[:5], 5, None),
    (40_003, SMALL[:5], 2, {"sort_digit_bits": 11}),  # a last group of one
    (3001, SMALL[:3], 1, None),
    (20_001, WIDE, 3, None),
    (40_001, WIDE, 3, {"sort_digit_bits": 10}),
])
def test_calls_in_a_row_match_frames(n, sizes, group, tune):
    import torch
    from paper_2605_04844_gb300 import _native as N
    from paper_2605_04844_gb300 import rasterizer as R
    sd = to_device(synth.scene_ball(n, 9 + n, radius=3.0, deg=1))
    s = R.scene_struct(sd)
    bg = (0.1, 0.2, 0.3)
    b = R.calibrated_batch(sd, cameras(sizes, 0.0), group=group, headroom=1.4)
    for turn in (0.0, 0.9):
        cams = cameras(sizes, turn)
        ca = R.camera_array(cams)
        b.render(s, ca, "quadbox", tune=tune, bg=bg)
        dL = torch.randn(b.images.shape, generator=torch.Generator("cuda").manual_seed(3), device="cuda")
        gb, gsb = grads_of(sd)
        b.backward(s, ca, dL, gsb, bg=bg)
        torch.cuda.synchronize()
        b.check()
        gf, gsf = grads_of(sd)
        for k, c in enumerate(cams):
            img, fr = R.forward(sd, c, "quadbox", bg=bg)
            assert torch.equal(b.image(k), img), (turn, k)
            N.qb_render_bwd(fr.frame, s, R.camera_struct(c), bg, b.image(k, dL).contiguous(), gsf, None)
        torch.cuda.synchronize()
        for k in KEYS:
            a, r = gb[k].double(), gf[k].double()
            assert (torch.linalg.norm(a - r) / torch.linalg.norm(r)).item() <= 1e-5, (turn, k)

"""The chain to the scene parameters of one camera's view runs over the list
of Gaussians with a screen-space gradient: every one of them exactly once, at
the edges of the spans the list is made from (512 Gaussians) and for sums that
are 16-byte aligned and not."""
import numpy as np
import pytest

from paper_2605_04844_gb300 import synth

from gpu_util import to_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 511, 512, 513, 1024, 1537, 5003])
@pytest.mark.parametrize("offset", [0, 1])
def test_every_gaussian_with_a_screen_gradient_once(n, offset):
    import torch
    from paper_2605_04844_gb300 import _native as N
    from paper_2605_04844_gb300 import rasterizer as R
    cam = synth.pinhole(200, 120)
    scene = synth.scene_uniform(n, 40 + n, cam, depth=(2.0, 6.0))
    scene["opacities"][:] = np.clip(scene["opacities"], -3.0, 3.0)
    sd = to_device(scene)
    _, fr = R.forward(sd, cam, "quadbox", bg=(0.1, 0.2, 0.3))
    dL = torch.randn((3, 120, 200), generator=torch.Generator().manual_seed(n)).cuda()
    g = {k: torch.zeros_like(v) for k, v in sd.items() if isinstance(v, torch.Tensor)}
    gs = N.QbSceneGrads()
    for k in ("means", "scales", "quats", "opacities", "sh"):
        setattr(gs, k, g[k].data_ptr())
    sums = torch.zeros(9 * n + offset, dtype=torch.float64, device="cuda")[offset:]
    N.qb_render_bwd(fr.frame, R.scene_struct(sd), R.camera_struct(cam), (0.1, 0.2, 0.3), dL, gs, sums, fr.stream)
    torch.cuda.synchronize()
    s = sums.cpu().numpy().reshape(n, 9)
    assert (s != 0).any()
    # dL/dlogit = dL/do o (1 - o): o within 3 * 2^-24 and 1 - o >= 0.047, so 1e-5
    o = 1.0 / (1.0 + np.exp(-scene["opacities"].astype(np.float64).reshape(n)))
    np.testing.assert_allclose(g["opacities"].cpu().numpy().reshape(n), s[:, 5] * o * (1 - o), rtol=1e-5, atol=1e-30)
    moved = np.zeros(n, bool)
    for k in ("means", "scales", "quats", "opacities", "sh"):
        moved |= (g[k].cpu().numpy().reshape(n, -1) != 0).any(axis=1)
    np.testing.assert_array_equal(moved, (s != 0).any(axis=1))

"""The counted render's second count at its threshold: an exponent equal to
-logf(255 o) - 0.001 (float32 operations) passes the power test, the next
lower float does not, for every opacity."""
import numpy as np
import pytest

from paper_2605_04844_gb300 import synth

pytestmark = pytest.mark.gpu


def test_exponents_at_the_threshold_are_counted():
    import torch
    from paper_2605_04844_gb300 import _native as N
    from paper_2605_04844_gb300 import rasterizer as R
    T = 32  # T x T tiles, one Gaussian in the middle of each
    n, W = T * T, 16 * T
    cam = synth.pinhole(W, W)
    c = 16.0 * np.arange(T) + 8.0
    px, py = (v.ravel() for v in np.meshgrid(c, c))
    z = 2.0
    means = np.stack([(px - cam["cx"]) * z / cam["fx"], (py - cam["cy"]) * z / cam["fy"], np.full(n, z)], 1)
    dev = lambda a: torch.tensor(np.ascontiguousarray(a), dtype=torch.float32, device="cuda")
    scene = {"means": dev(means), "scales": dev(np.full((n, 3), 0.1 * z / cam["fx"])),
             "quats": dev(np.tile([1.0, 0, 0, 0], (n, 1))), "opacities": dev(np.linspace(0.02, 0.97, n)),
             "sh": dev(np.full((n, 1, 3), 0.1)), "sh_degree": 0, "raw": 0}
    img, fr = R.forward(scene, cam, "quadbox")
    a = fr.arrays()
    assert fr.n_pairs == n  # a tile each
    a["xy"].copy_(a["xy"].round())
    o = a["conic_o"][:, 3].clone()
    t = -torch.log(torch.tensor(255.0, device="cuda") * o) - 1e-3
    below = torch.nextafter(t, torch.full_like(t, -np.inf))
    # power = -(a / 2)(dx^2 + dy^2): t at the four neighbours of the centre
    for power, per_gaussian in ((t, 5), (below, 1)):
        a["conic_o"][:, 0] = -2.0 * power
        a["conic_o"][:, 1] = 0.0
        a["conic_o"][:, 2] = -2.0 * power
        cnt = torch.zeros(2, dtype=torch.int64, device="cuda")
        N.qb_render_fwd_counted(fr.frame, None, torch.empty_like(img), cnt)
        assert cnt.tolist() == [256 * n, per_gaussian * n]

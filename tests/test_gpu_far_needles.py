"""Needles whose mean lies far outside the image (10^5 to 10^8 pixels) and whose
long axis crosses it: every pixel that the render's own float32 exponent accepts
is composited, and no other.  The ellipse test ahead of the pixels must not
drop an entry that its rounding cannot tell from one that misses the tile."""
import numpy as np
import pytest

from paper_2605_04844_gb300 import synth

from gpu_util import to_device

pytestmark = pytest.mark.gpu

f32 = np.float32


def fma(a, b, c):
    """float32 fma by float64 (the product of two float32 is exact there)."""
    return (np.asarray(a, np.float64) * np.asarray(b, np.float64) + np.asarray(c, np.float64)).astype(f32)


@pytest.mark.parametrize("distance", [1e5, 1e7, 3e7, 1e8])
def test_far_needles_reach_their_pixels(distance):
    import torch
    from paper_2605_04844_gb300 import _native as N
    from paper_2605_04844_gb300 import rasterizer as R
    W = H = 64
    cam = synth.pinhole(W, H)
    rng = np.random.default_rng(int(distance))
    checked = 0
    for k in range(120):
        th = rng.uniform(0.1, 1.4) + 0.5 * np.pi * rng.integers(0, 4)
        u = np.array([np.cos(th), np.sin(th)])
        sig, thin = distance * rng.uniform(0.5, 2.0), rng.uniform(0.2, 2.5)  # pixels
        mu = distance * u + rng.uniform(-1, 1) * thin * np.array([-u[1], u[0]])
        scene = {"means": np.array([[mu[0] / cam["fx"], mu[1] / cam["fy"], 1.0]]),
                 "scales": np.log([[sig / cam["fx"], thin / cam["fx"], 1e-3]]),
                 "quats": np.array([[np.cos(th / 2), 0.0, 0.0, np.sin(th / 2)]]),
                 "opacities": np.array([rng.uniform(-2.0, 2.0)]), "sh": np.full((1, 1, 3), 0.5),
                 "sh_degree": 0, "raw": 1}
        img, fr = R.forward(to_device(scene), cam, "aabb3s")
        torch.cuda.synchronize()
        A = {k: v.cpu().numpy() for k, v in fr.arrays().items()}
        if A["counts"][0] == 0:
            continue
        # the terms of the exact form, behind the means in the frame's workspace
        arr = N.qb_frame_arrays_get(fr.frame)
        shape = fr._view(arr.xy + 256, torch.float32, (1, 2)).cpu().numpy()[0]
        (mx, my), (a, b, c, o) = A["xy"][0], A["conic_o"][0]
        assert shape[1] != 0 and max(abs(mx), abs(my)) > 0.3 * distance
        px, py = np.meshgrid(np.arange(W, dtype=f32), np.arange(H, dtype=f32))
        dx, dy = f32(mx) - px, f32(my) - py
        v = fma(shape[0], dy, dx)
        power = fma(f32(-0.5) * a * v, v, f32(shape[1]) * dy * dy).astype(np.float64)
        edge = -np.log(255.0 * o)  # alpha = 1/255
        tiles = (A["ranges"].reshape(-1, 2)[:, 1] > A["ranges"].reshape(-1, 2)[:, 0]).reshape(H // 16, W // 16)
        listed = np.kron(tiles, np.ones((16, 16), bool))
        want = listed & (power > edge + 1e-3)
        unsure = np.abs(power - edge) <= 1e-3
        got = A["n_contrib"] > 0
        assert not np.any((got != want) & ~unsure), f"{int(((got != want) & ~unsure).sum())} pixels of needle {k}"
        checked += int(want.any())
    assert checked > 20

"""The Adam kernel's vector and scalar forms at the sizes where their
remainders lie, and the single-camera backward's list of nonzero sums against
the several-camera form, which takes every Gaussian in turn."""
import numpy as np
import pytest

from paper_2605_04844_gb300 import synth

from gpu_util import to_device

pytestmark = pytest.mark.gpu

KEYS = ("means", "scales", "quats", "opacities", "sh")


@pytest.mark.parametrize("n", [1, 3, 4, 7, 1023, 1_000_003])
@pytest.mark.parametrize("offset", [0, 1])
def test_adam_vector_and_scalar_forms(n, offset):
    """offset 1: arrays that are not 16-byte aligned take the scalar form."""
    import torch
    from paper_2605_04844_gb300 import _native as N
    g = torch.Generator("cuda").manual_seed(n)
    buf = [torch.randn(n + 1, generator=g, device="cuda") for _ in range(4)]
    buf[3].abs_()
    p, gr, m, v = (b[offset:offset + n] for b in buf)
    P, G, M, V = (t.double() for t in (p, gr, m, v))
    tail = [b.clone() for b in buf]
    lr, b1, b2, eps, t = 1e-2, 0.9, 0.999, 1e-8, 7
    N.qb_adam_step(p, gr, m, v, lr, b1, b2, eps, t)
    M, V = b1 * M + (1 - b1) * G, b2 * V + (1 - b2) * G * G
    want = P - lr * (M / (1 - b1 ** t)) / ((V / (1 - b2 ** t)).sqrt() + eps)
    # float32 rounding of a few operations, and of 1 - b2^t (2e-3 here, from powf: 2^-24 / 7e-3)
    assert torch.allclose(m.double(), M, rtol=1e-5, atol=1e-6)
    assert torch.allclose(v.double(), V, rtol=1e-4, atol=1e-6)
    assert torch.allclose(p.double(), want, rtol=1e-5, atol=1e-5)
    for b, old in zip(buf, tail):  # nothing outside the arrays
        outside = torch.ones(n + 1, dtype=torch.bool, device="cuda")
        outside[offset:offset + n] = False
        assert torch.equal(b[outside], old[outside])


def _grads(sd):
    import torch
    from paper_2605_04844_gb300 import _native as N
    g = {k: torch.zeros_like(sd[k]) for k in KEYS}
    gs = N.QbSceneGrads()
    for k in KEYS:
        setattr(gs, k, g[k].data_ptr())
    return g, gs


@pytest.mark.parametrize("n", [1, 511, 512, 513, 5003])
@pytest.mark.parametrize("deg", [0, 1, 2, 3])
@pytest.mark.parametrize("nan_at", [None, 0])
def test_listed_backward_matches_the_per_gaussian_form(n, deg, nan_at):
    """Two equal cameras give twice the gradient of one (the sums of equal
    terms double exactly; the two forms may contract products differently).  A
    Gaussian whose colour is not finite keeps its NaN direction gradient."""
    import torch
    from paper_2605_04844_gb300 import _native as N
    from paper_2605_04844_gb300 import rasterizer as R
    cam = synth.pinhole(70, 50)
    scene = synth.scene_uniform(n, 3 + n, cam, deg=deg)
    if nan_at is not None:
        scene["sh"][nan_at, -1, 1] = np.nan
        scene["opacities"][nan_at] = -5.0  # faint, visible
        scene["means"][nan_at] = [1e3, 0.0, 2.0]  # beyond the image: no pixel composites it
    sd = to_device(scene)
    s, c = R.scene_struct(sd), R.camera_struct(cam)
    img, fr = R.forward(sd, cam, "quadbox")
    dL = torch.randn(img.shape, generator=torch.Generator("cuda").manual_seed(1), device="cuda")
    g1, gs1 = _grads(sd)
    N.qb_render_bwd(fr.frame, s, c, None, dL, gs1)
    b = R.calibrated_batch(sd, [cam, cam], group=2)
    b.render(s, R.camera_array([cam, cam]), "quadbox")
    g2, gs2 = _grads(sd)
    b.backward(s, R.camera_array([cam, cam]), torch.cat([dL.reshape(-1)] * 2), gs2)
    torch.cuda.synchronize()
    for k in KEYS:
        x, y = g1[k].double(), g2[k].double()
        assert torch.equal(torch.isnan(x), torch.isnan(y))
        if nan_at is not None and k == "means" and deg > 0:
            assert torch.isnan(x[nan_at]).all()
        x, y = torch.nan_to_num(2 * x), torch.nan_to_num(y)
        assert torch.linalg.norm(x - y) <= 1e-5 * torch.linalg.norm(x) + 1e-30, k

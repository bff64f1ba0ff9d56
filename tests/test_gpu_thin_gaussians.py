"""Thin Gaussians (aspect 10 : 1 to 2000 : 1, at every angle) against the
oracle: the half-tile ellipse test of elongated conics must keep every entry
that a pixel composites."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2605_04844_gb300 import synth

from gpu_util import f64, image_parity, run_forward

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("long_axis,thin", [(0.2, -6.0), (0.8, -6.5), (1.6, -5.0)])
@pytest.mark.parametrize("mode", ["quadbox", "aabb3s+noclamp"])
def test_thin_gaussians_match_the_oracle(long_axis, thin, mode):
    W, H = 330, 210
    cam = synth.pinhole(W, H)
    rng = np.random.default_rng(int(100 * long_axis))
    scene = synth.scene_uniform(700, 8, cam, depth=(2.0, 6.0))
    scene["scales"][:] = rng.normal(thin, 0.3, scene["scales"].shape)
    scene["scales"][np.arange(700), rng.integers(0, 3, 700)] = rng.normal(np.log(long_axis), 0.4, 700)
    img, fr, A = run_forward(scene, cam, mode, bg=(0.1, 0.2, 0.3))
    assert (A["meta"] & 1).sum() > 600
    name, clamp = mode.split("+")[0], "+" not in mode
    ref = O.image(f64(scene), cam, O.QUADBOX if name == "quadbox" else O.AABB3S, clamp3s=clamp, bg=(0.1, 0.2, 0.3))
    ok, st = image_parity(img, ref)
    assert ok, st

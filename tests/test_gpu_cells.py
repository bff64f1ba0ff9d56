"""The depth-first binning through cells of 8 x 4 tiles against the full-key
sort of all pairs: the same sorted values and ranges at the sizes where the
cells can go wrong (one cell exactly, one pixel more, cells cut by the image's
edge, ids sorted in one, two and three passes, more cells than a block's
shared-memory histogram holds) and for every traversal, odd counts among them."""
import numpy as np
import pytest

from paper_2605_04844_gb300 import synth

from gpu_util import to_device

pytestmark = pytest.mark.gpu


def both_paths(scene, cam, mode, digit_bits=8):
    import torch
    from paper_2605_04844_gb300 import rasterizer as R
    sd = to_device(scene)
    out = []
    for sort_mode in ("depth_first", "full_key"):
        img, fr = R.forward(sd, cam, mode, bg=(0.3, 0.2, 0.1), sort_mode=sort_mode, digit_bits=digit_bits)
        torch.cuda.synchronize()
        fr.check()
        a = fr.arrays()
        out.append((fr.n_pairs, a["vals"].cpu().numpy(), a["ranges"].cpu().numpy(), img.cpu().numpy()))
    (pa, va, ra, ia), (pb, vb, rb, ib) = out
    assert pa == pb
    np.testing.assert_array_equal(va, vb)
    np.testing.assert_array_equal(ra, rb)
    np.testing.assert_array_equal(ia, ib)
    return pa


@pytest.mark.parametrize("W,H", [(128, 64), (129, 65), (127, 1), (1, 300), (1000, 520), (2560, 1440), (3840, 2160),
                                 (8208, 4096)])
@pytest.mark.parametrize("mode", ["quadbox", "aabb3s"])
def test_cells_at_the_edges_of_their_sizes(W, H, mode):
    cam = synth.pinhole(W, H)
    scene = synth.scene_blobs(9_001, 31 + W, cam, deg=0)
    assert both_paths(scene, cam, mode) > 0


@pytest.mark.parametrize("mode", ["adr", "quadbox_naive", "dualbox", "quadbox+noclamp", "aabb3s"])
@pytest.mark.parametrize("digit_bits", [8, 11])
def test_cells_of_every_traversal(mode, digit_bits):
    cam = synth.pinhole(2000, 1100)
    both_paths(synth.scene_blobs(30_003, 77, cam, deg=0), cam, mode, digit_bits)


def test_crowded_cells_and_gaussians_that_fill_the_image():
    """Rows of many entries in few cells (a small image), and Gaussians whose
    boxes cover every cell of a large one."""
    cam = synth.pinhole(200, 100)
    both_paths(synth.scene_uniform(300_001, 5, cam), cam, "quadbox")
    cam = synth.pinhole(3000, 2000)
    scene = synth.scene_uniform(400, 6, cam, depth=(1.0, 3.0), logscale=(0.5, 0.6))
    assert both_paths(scene, cam, "quadbox") > 1_000_000

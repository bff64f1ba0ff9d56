"""A look-back that runs out, in each of the binning's sorts and in its count
scan: the frame reports TIMEOUT, its lists are empty (nothing is gathered
through an order with gaps or through offsets that do not belong together), it
renders the background, and it works again once the error is taken.  No wait
hangs and no GPU fault is involved: the test-only word (err_flags[1]) ends one
block's walk as a wait that ran out would."""
import numpy as np
import pytest

from paper_2605_04844_gb300 import synth

from gpu_util import to_device

pytestmark = pytest.mark.gpu

POLLS, SCAN, KEYED = 64, 1 << 29, 1 << 30


def one_tile_gaussians(n, cam):
    """Gaussians of a fraction of a pixel: one tile each, so that any n entries
    have the same total of tiles."""
    scene = synth.scene_uniform(n, 11, cam, depth=(2.0, 3.0))
    scene["scales"][:] = np.log(0.1 * 2.0 / cam["fx"])
    return scene


# word, n, image, sort mode: the pass or scan that the word ends
CASES = [
    (POLLS, 20_000, (256, 256), "depth_first"),        # the cell sort's only pass
    (POLLS, 20_000, (2560, 1440), "depth_first"),      # ... its second of two
    (KEYED, 20_000, (2560, 1440), "depth_first"),      # ... its first of two
    (KEYED, 70_001, (256, 256), "depth_first"),        # the depth order's passes
    (KEYED, 20_000, (256, 256), "full_key"),           # the pair sort's passes
    (SCAN, 70_001, (256, 256), "depth_first"),
    (SCAN, 20_000, (256, 256), "full_key"),
    (KEYED | SCAN, 70_001, (256, 256), "depth_first"),
]


@pytest.mark.parametrize("word,n,size,sort_mode", CASES)
@pytest.mark.parametrize("mode", ["quadbox", "quadbox_naive"])
@pytest.mark.parametrize("sync", [True, False])
def test_a_timed_out_frame_is_empty_and_recovers(word, n, size, sort_mode, mode, sync):
    import torch
    from paper_2605_04844_gb300 import _native as N
    from paper_2605_04844_gb300 import rasterizer as R
    W, H = size
    cam = synth.pinhole(W, H)
    sd = to_device(one_tile_gaussians(n, cam))
    s, c = R.scene_struct(sd), R.camera_struct(cam)
    bg = (0.25, 0.5, 0.75)
    # the buffers hold this scene's own lists when the wait runs out
    ref, fr = R.forward(sd, cam, mode, bg=bg, sort_mode=sort_mode)
    fr.check()
    assert fr.n_pairs > 8192
    want = {k: fr.arrays()[k].clone() for k in ("vals", "ranges")}
    P = fr.n_pairs
    flags = fr.arrays()["err_flags"]
    flags[1] = word
    fr.preprocess(s, c, mode)
    fr.bin_emit(sync=sync)
    fr.sort()
    img = fr.render(bg)
    torch.cuda.synchronize()
    assert int(fr.arrays(n_pairs=0)["ranges"].abs().max().item()) == 0
    for ch in range(3):
        assert torch.equal(img[ch], torch.full_like(img[ch], bg[ch]))
    with pytest.raises(N.QbError) as ei:
        fr.check()
    assert ei.value.status == N.QB_ERR_TIMEOUT

    flags[1] = 0
    fr.preprocess(s, c, mode)
    fr.bin_emit(sync=sync)
    fr.sort()
    img = fr.render(bg)
    torch.cuda.synchronize()
    fr.check()
    a = fr.arrays(n_pairs=P)
    for k, v in want.items():
        assert torch.equal(a[k], v), k
    assert torch.equal(img, ref)

"""qb_bin_emit called again without a new qb_preprocess (a caller that reads the
pair count first and emits later, a captured graph of the later stages replayed):
every call gives the same order, pairs and image, on both sides of the limit
between the two depth sorts."""
import numpy as np
import pytest

from paper_2605_04844_gb300 import synth

from gpu_util import to_device

pytestmark = pytest.mark.gpu

KEYS = ("depth_order", "offsets", "vals", "ranges")


@pytest.mark.parametrize("n", [7, 3000, 32_768, 32_769])
@pytest.mark.parametrize("sort_mode", ["depth_first", "full_key"])
def test_emit_again_gives_the_same_order(n, sort_mode):
    import torch
    from paper_2605_04844_gb300 import rasterizer as R
    cam = synth.pinhole(300, 200)
    sd = to_device(synth.scene_uniform(n, 17 + n, cam, depth=(0.1, 6.0)))
    img, fr = R.forward(sd, cam, "quadbox", bg=(0.1, 0.2, 0.3), sort_mode=sort_mode)
    keys = KEYS if sort_mode == "depth_first" else KEYS[1:]
    first = {k: fr.arrays()[k].clone() for k in keys}
    P = fr.n_pairs
    for sync in (True, False):
        fr.bin_emit(sync=sync)
        fr.sort()
        again = fr.render((0.1, 0.2, 0.3))
        torch.cuda.synchronize()
        fr.check()
        a = fr.arrays(n_pairs=P)
        for k in keys:
            np.testing.assert_array_equal(a[k].cpu().numpy(), first[k].cpu().numpy(), err_msg=k)
        assert torch.equal(again, img)


def test_a_graph_of_the_later_stages_replays():
    import torch
    from paper_2605_04844_gb300 import rasterizer as R
    cam = synth.pinhole(256, 256)
    sd = to_device(synth.scene_uniform(5000, 3, cam, depth=(0.1, 6.0)))
    img, fr = R.forward(sd, cam, "quadbox")
    out = torch.empty_like(img)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        fr.bin_emit(sync=False)
        fr.sort()
        fr.render(None, out)
    for _ in range(3):
        out.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, img)
    fr.check()

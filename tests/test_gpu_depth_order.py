"""The depth order of few Gaussians (one cluster, in shared memory) at the
sizes where its shares of keys per block and per thread change, against
numpy's stable sort; the counts' prefixes in that order; and the pairs of the
sizes on both sides of the limit against the full-key path."""
import numpy as np
import pytest

from paper_2605_04844_gb300 import synth

from gpu_util import to_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 32, 33, 255, 257, 8191, 8192, 8193, 16384, 16385, 32767, 32768, 32769])
@pytest.mark.parametrize("ties", [False, True])
def test_depth_order_and_prefixes(n, ties):
    import torch
    from paper_2605_04844_gb300 import rasterizer as R
    cam = synth.pinhole(400, 300)
    scene = synth.scene_uniform(n, 90 + n, cam, depth=(0.1, 6.0))  # some before the near plane
    if ties:  # few distinct depths: order by index within one
        scene["means"][:, 2] = np.round(scene["means"][:, 2] * 4) / 4
    sd = to_device(scene)
    _, fr = R.forward(sd, cam, "quadbox")
    torch.cuda.synchronize()
    fr.check()
    A = {k: v.cpu().numpy() for k, v in fr.arrays().items() if k in ("rgbd", "counts", "depth_order", "offsets", "vals")}
    d = A["rgbd"][:, 3].astype(np.float32).view(np.uint32) & np.uint32(0x7FFFFFFF)
    key = np.where(A["counts"] > 0, d, np.uint32(0x7FFFFFFF))
    order = np.argsort(key, kind="stable")
    np.testing.assert_array_equal(A["depth_order"].view(np.uint32), order.astype(np.uint32))
    c = A["counts"].astype(np.int64)[order]
    np.testing.assert_array_equal(A["offsets"].astype(np.int64), np.cumsum(c) - c)
    assert fr.n_pairs == int(c.sum())
    _, full = R.forward(sd, cam, "quadbox", sort_mode="full_key")
    np.testing.assert_array_equal(A["vals"], full.arrays()["vals"].cpu().numpy())


@pytest.mark.parametrize("n", [24_575, 24_576, 24_577])
def test_depth_order_around_three_keys_per_thread(n):
    test_depth_order_and_prefixes(n, False)


def test_overflow_of_a_small_scene_writes_nothing():
    import torch
    from paper_2605_04844_gb300 import _native as N
    from paper_2605_04844_gb300 import rasterizer as R
    cam = synth.pinhole(128, 128)
    sd = to_device(synth.scene_uniform(3000, 4, cam))
    fr = R.Frame(3000, 128, 128, pair_capacity=500)
    fr.preprocess(R.scene_struct(sd), R.camera_struct(cam), "quadbox")
    fr.bin_emit(sync=False)
    fr.sort()
    img = fr.render((0.25, 0.5, 0.75))
    torch.cuda.synchronize()
    with pytest.raises(N.QbCapacityError):
        fr.check()
    assert torch.equal(img[1], torch.full_like(img[1], 0.5))

"""Device memory of frames and batches: no configuration takes more than these
figures, which callers have sized their memory by (a frame's may move by its
scan table, 0.05 %)."""
import pytest

from paper_2605_04844_gb300 import _native as N

FRAMES = [  # n, width, height, pair capacity, bytes
    (10000, 256, 256, 65536, 5590016),
    (200000, 1001, 701, 5000000, 218521856),
    (1000000, 1920, 1080, 38000000, 1487996416),
    (3000000, 2560, 1440, 60000000, 2819012096),
    (1000000, 3840, 2160, 140000000, 5121127680),
    (1000000, 1920, 1080, 1073741824, 34647896832),
]
BATCHES = [  # n, cameras, width, height, group, pair capacity, bytes
    (1000000, 16, 1920, 1080, 16, 35000000, 8586120704),
    (200000, 5, 1264, 832, 5, 10000000, 1143740672),
    (1000000, 64, 1920, 1080, 16, 35000000, 23607649792),
    (1000000, 16, 1920, 1080, 16, 8000000, 5128485376),
    (50000, 8, 640, 480, 8, 400000, 159432448),
    (1000000, 4, 1920, 1080, 1, 40000000, 4031070208),
    (1000000, 16, 2560, 1440, 16, 60000000, 12098271744),
    (1000000, 16, 1920, 1080, 16, 1073741824, 141609990656),
    (3000000, 32, 1920, 1080, 16, 100000000, 38221403136),
    (1000, 3, 64, 64, 3, 65536, 5954816),
]


@pytest.mark.parametrize("n,W,H,cap,most", FRAMES)
def test_frame_workspace(n, W, H, cap, most):
    assert 0 < N.qb_frame_workspace_bytes(n, W, H, cap) <= 1.0005 * most


@pytest.mark.parametrize("n,cams,W,H,group,cap,most", BATCHES)
def test_batch_workspace(n, cams, W, H, group, cap, most):
    assert 0 < N.qb_batch_workspace_bytes(n, [W] * cams, [H] * cams, group, cap) <= most

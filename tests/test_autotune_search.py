"""The autotuner times only parameters that change what is launched: on
timings that fall from call to call (the last candidate always looks best),
render_batch, which has no effect, keeps its default and is never varied."""
import itertools

import pytest

from paper_2605_04844_gb300 import autotune as T


class FakeFrame:
    def __init__(self):
        self.tunings = []
        self.ws = type("W", (), {"device": "cpu"})

    def set_tuning(self, **kw):
        self.tunings.append(kw)

    def preprocess(self, *a):
        pass

    bin_emit = sort = render = check = lambda self, *a, **k: None


class FakeBatch:
    n, n_cams, group, widths, heights = 10, 2, 2, [8, 8], [8, 8]

    def __init__(self):
        self.cands = []

    def render(self, scene, cams, mode, cand):
        self.cands.append(cand)

    def check(self):
        pass


@pytest.fixture
def fake(monkeypatch):
    fall = itertools.count(1000, -1)

    def time(fn, reps):
        fn()
        return float(next(fall))

    monkeypatch.setattr(T, "_time", time)
    monkeypatch.setattr(T.torch.cuda, "get_device_name", lambda: "none")
    for f in ("scene_struct", "camera_struct", "camera_array"):
        monkeypatch.setattr(T.R, f, lambda x: x)
    return monkeypatch


def test_frame_search(fake):
    fr = FakeFrame()
    fake.setattr(T.R, "forward", lambda *a: (None, fr))
    scene = {"means": type("M", (), {"shape": (10, 3)})}
    res = T.tune_frame(scene, {"width": 8, "height": 8}, use_cache=False)
    assert res["digit_bits"] == 11 and res["render_batch"] == 128
    assert not any("render_batch" in t for t in fr.tunings)


def test_batch_search(fake):
    b = FakeBatch()
    res = T.tune_batch(b, None, [None, None], use_cache=False)
    assert res["tune"] == {"sort_digit_bits": 11, "render_batch": 128, "tiles_per_fetch": 4, "blocks_per_sm": 4}
    assert {c["render_batch"] for c in b.cands} == {128}
    assert len({tuple(sorted(c.items())) for c in b.cands}) >= 7

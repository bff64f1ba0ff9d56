"""What camera_struct takes as a camera's arrays, and what it refuses: the same
values from every form that a tensor can be made of."""
import numpy as np
import pytest
import torch

from paper_2605_04844_gb300 import rasterizer as R
from paper_2605_04844_gb300 import synth

FORMS = [
    lambda a: a, lambda a: a.astype(np.float64), lambda a: a.tolist(), lambda a: torch.from_numpy(a),
    lambda a: np.asfortranarray(a), lambda a: a.astype(np.float16), np.matrix, np.ma.masked_array,
    lambda a: np.repeat(a, 2, axis=-1)[..., ::2],
]


@pytest.mark.parametrize("form", FORMS)
def test_forms_of_the_camera_arrays(form):
    cam = synth.pinhole(64, 48, viewmat=np.array([[0, 1, 0, 2.5], [-1, 0, 0, 0.5], [0, 0, 1, 3], [0, 0, 0, 1.0]]))
    c = R.camera_struct(dict(cam, viewmat=form(cam["viewmat"]), campos=form(cam["campos"])))
    assert list(c.viewmat) == cam["viewmat"].ravel().tolist()
    assert list(c.campos) == cam["campos"].tolist()


@pytest.mark.parametrize("bad", [lambda a: a[:3], lambda a: a[::-1], lambda a: a.astype(">f4"), lambda a: None])
def test_refused_forms(bad):
    cam = synth.pinhole(64, 48)
    with pytest.raises(Exception):
        R.camera_struct(dict(cam, viewmat=bad(cam["viewmat"])))

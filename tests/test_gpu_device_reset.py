"""A cudaDeviceReset between frames leaves nothing stale behind: not the host
word of the pair count, not the kernels' shared-memory limits (in a process of
its own, without torch)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

RESET = r"""
import ctypes, sys
import numpy as np
from paper_2605_04844_gb300 import _native as N, synth
rt = ctypes.CDLL(sys.argv[1])
L = N.load(build_if_missing=False)
def alloc(nbytes):
    p = ctypes.c_void_p()
    assert rt.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(max(nbytes, 256))) == 0
    return p
def count(n, deg):
    cam = synth.pinhole(64, 64)
    sc = synth.scene_blobs(n, 5, cam, deg=deg)
    s, c = N.QbScene(), N.QbCamera()
    for k in ("means", "scales", "quats", "opacities", "sh"):
        a = np.ascontiguousarray(sc[k], np.float32)
        p = alloc(a.nbytes)
        assert rt.cudaMemcpy(p, a.ctypes.data_as(ctypes.c_void_p), ctypes.c_size_t(a.nbytes), 1) == 0
        setattr(s, k, p.value)
    s.n, s.sh_degree, s.params_raw = n, deg, 1
    c.viewmat[:] = cam["viewmat"].ravel().tolist()
    c.campos[:] = cam["campos"].tolist()
    for k in ("fx", "fy", "cx", "cy", "tan_fovx", "tan_fovy", "znear"):
        setattr(c, k, float(cam[k]))
    c.width = c.height = 64
    nb = L.qb_frame_workspace_bytes(n, 64, 64, 1 << 16)
    f, P = N.QbFrame(), ctypes.c_uint64(0)
    N.check(L.qb_frame_init(ctypes.byref(f), n, 64, 64, 1 << 16, alloc(nb), nb, None))
    N.check(L.qb_preprocess(ctypes.byref(f), ctypes.byref(s), ctypes.byref(c), 1, None))
    N.check(L.qb_bin_emit(ctypes.byref(f), ctypes.byref(P), None))
    N.check(L.qb_sort(ctypes.byref(f), None))
    N.check(L.qb_render_fwd(ctypes.byref(f), None, alloc(3 * 64 * 64 * 4), None))
    assert rt.cudaDeviceSynchronize() == 0
    N.check(L.qb_frame_check(ctypes.byref(f), None))
    return P.value
before = [count(2000, 3), count(40000, 0)]
for _ in range(3):
    assert rt.cudaDeviceReset() == 0
    assert [count(2000, 3), count(40000, 0)] == before
print("same", before)
"""


def test_a_device_reset_leaves_nothing_stale():
    cudart = "/usr/local/cuda/lib64/libcudart.so"
    if not os.path.exists(cudart):
        pytest.skip("no shared CUDA runtime")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", RESET, cudart], cwd=root, capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and "same" in r.stdout, r.stdout + r.stderr

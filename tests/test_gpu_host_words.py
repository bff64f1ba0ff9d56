"""The host word that a synchronised qb_bin_emit reads the pair count from:
threads that call at the same time get their own counts, and a thread that ends
leaves another thread's graph capture alone."""
import os
import threading
import time

import pytest

from paper_2605_04844_gb300 import synth

from gpu_util import to_device

pytestmark = pytest.mark.gpu


def frame_of(n, W, H, stream=None):
    from paper_2605_04844_gb300 import rasterizer as R
    cam = synth.pinhole(W, H)
    sd = to_device(synth.scene_uniform(n, n, cam))
    fr = R.Frame(n, W, H, pair_capacity=1 << 20, stream=stream)
    fr.preprocess(R.scene_struct(sd), R.camera_struct(cam), "quadbox")
    return sd, fr


def test_threads_get_their_own_counts():
    import torch
    made = []
    for k in range(8):
        sd, fr = frame_of(500 + 700 * k, 160, 120)
        want = fr.bin_emit(sync=True)
        fr.stream = torch.cuda.Stream()
        made.append((sd, fr, want))
    assert len({w for _, _, w in made}) == len(made)
    torch.cuda.synchronize()
    bad = []

    def work(fr, want):
        for _ in range(200):
            if fr.bin_emit(sync=True) != want:
                bad.append(want)

    threads = [threading.Thread(target=work, args=(fr, w)) for _, fr, w in made]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad


def test_a_thread_that_ends_leaves_a_capture_alone():
    import torch
    go = threading.Event()
    ready = threading.Event()

    def work():
        sd, fr = frame_of(900, 96, 96)
        fr.bin_emit(sync=True)
        torch.cuda.synchronize()
        ready.set()
        go.wait()

    t = threading.Thread(target=work)
    t.start()
    ready.wait()
    task = f"/proc/self/task/{t.native_id}"
    x = torch.zeros(64, device="cuda")
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode="global"):
        x += 1.0
        go.set()
        t.join()
        for _ in range(500):  # until the thread itself is gone
            if not os.path.exists(task):
                break
            time.sleep(0.01)
        x += 1.0
    g.replay()
    torch.cuda.synchronize()
    assert float(x[0]) == 2.0

"""A batch leaves the caller's more urgent streams ahead of its own launches."""
import ctypes
import threading
import time

import pytest

from gpu_common import need_gpu, to_dev, torch
from paper_1810_02821_gb300 import build, synth, wf

pytestmark = pytest.mark.gpu


def test_batch_on_a_background_stream_does_not_overtake_an_urgent_one():
    """A batch of about twenty rounds of 128 x 128 solves on a stream of the least priority, and a small kernel on one of the
    greatest priority that torch gives, launched a third of the way through: it runs as soon as a CTA of the batch ends, not
    after the batch's last CTA has started."""
    need_gpu()
    build.build()
    lib = wf.load_library()
    n = 6000
    p = synth.make_problem(128, seed=1, mask_frac=0.1, slope=-3.0, k0=1.0 / 16)
    dev = to_dev(p)
    out = torch.empty(n, 128, 128, device="cuda")
    items = wf._batch_items([wf.BatchImage(*dev, out_wf=out[i]) for i in range(n)], 0)
    opts = wf._batch_opts()
    background, urgent = torch.cuda.Stream(priority=0), torch.cuda.Stream(priority=-3)
    x = torch.zeros(64, device="cuda")

    def run():
        assert lib.wf_batch_run(items, n, ctypes.byref(opts), ctypes.c_void_p(background.cuda_stream)) == 0

    def small():
        with torch.cuda.stream(urgent):
            x.add_(1.0)
        urgent.synchronize()

    run(), small()  # warm up
    torch.cuda.synchronize()
    t = time.perf_counter()
    run()
    whole = time.perf_counter() - t
    share = []
    for _ in range(3):
        th = threading.Thread(target=run)
        th.start()
        time.sleep(whole / 3)
        t0 = time.perf_counter()
        small()
        t1 = time.perf_counter()
        th.join()
        t2 = time.perf_counter()
        share.append((t1 - t0) / (t2 - t0))  # of the batch's remaining time
    print(f"batch {whole * 1e3:.1f} ms, share of the remaining time waited: {share}")
    assert sorted(share)[1] < 0.5

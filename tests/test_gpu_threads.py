"""Handles of several threads at once, each on a stream of its own, from the library's first calls on a device on: every thread gets what
a thread alone gets."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2010_16165_b200 import workloads as wl
from test_gpu_parity import Gpu

pytestmark = pytest.mark.gpu


def test_threads_with_handles_of_their_own():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2010_16165_b200 import binding as B
    B.lib()
    loads = [wl.tiny_cifar(widths=(16, 32, 64), in_hw=32, batch=3, n_per_stage=1, p=0.3), wl.tiny_cifar(in_hw=24, batch=9, p=0.3),
             wl.tiny_imagenet_basic(batch=2, p=0.3), wl.tiny_imagenet_basic(widths=(32, 64, 96), in_hw=48, batch=3, p=0.3)] * 2
    got, failed = [None] * len(loads), []
    begin = threading.Barrier(len(loads))

    def work(i):
        try:
            begin.wait()
            g = Gpu(B, loads[i], B.FP_COMPUTE_BF16_TC)
            st = torch.cuda.Stream()
            B.fp_prune(g.h, loads[i].ratios)
            got[i] = [g.forward(loads[i].x, st) for _ in range(4)]
            g.close()
        except Exception as e:                                       # noqa: BLE001 - reported by the main thread
            failed.append(repr(e))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(loads))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed
    for i, w in enumerate(loads):
        g = Gpu(B, w, B.FP_COMPUTE_BF16_TC)
        try:
            B.fp_prune(g.h, w.ratios)
            want = g.forward(w.x)
        finally:
            g.close()
        for out in got[i]:
            np.testing.assert_array_equal(out, want)

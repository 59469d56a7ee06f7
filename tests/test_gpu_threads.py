"""Calls from threads that come and go: a thread that used the library leaves
nothing behind whose release would disturb the others."""
import os
import threading
import time

import pytest

pytestmark = pytest.mark.gpu

C4 = [(0, 1), (1, 2), (2, 3), (3, 0)]


@pytest.fixture(scope="module")
def tc():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_08975_gb300 import _build
    _build.build()
    from paper_2409_08975_gb300 import tc as tcmod
    tcmod.lib()
    return tcmod


def test_a_thread_may_end_while_another_captures(tc):
    # in the global capture mode an allocation or release of any thread that
    # could wait for the device ends the capture in an error
    import torch
    from paper_2409_08975_gb300 import synth
    c = synth.scaled_mid(3000, 60_000, seed=21)
    dev = lambda a, dt: torch.from_numpy(a).to(device="cuda", dtype=dt)  # noqa: E731
    g = tc.tc_build_temporal_csr(c["n"], dev(c["src"], torch.int32), dev(c["dst"], torch.int32), dev(c["t"], torch.int64))
    mot, kept = tc.make_motif(C4), []
    called, leave = threading.Event(), threading.Event()

    def work():
        try:
            w = tc.tc_path_weights(g, mot, 3600)
            kept.append((w, tc.tc_sample_estimate(g, mot, 3600, w, 10_000, 1)))
        finally:
            called.set()
            leave.wait(60)

    th = threading.Thread(target=work)
    th.start()
    assert called.wait(60) and kept
    task = "/proc/self/task/%d" % th.native_id
    x = torch.zeros(4, device="cuda")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, capture_error_mode="global"):
        x.add_(1)
        leave.set()
        th.join()
        for _ in range(1000):  # the thread's own storage is released after join returns
            if not os.path.exists(task):
                break
            time.sleep(0.01)
    assert not os.path.exists(task)
    x.zero_()
    graph.replay()
    assert x.tolist() == [1.0] * 4

"""Calls from one thread leave the others running."""
import threading
import time

import pytest

pytestmark = pytest.mark.gpu


def test_a_call_that_waits_for_room_in_the_queue_does_not_stop_other_threads():
    """Launches behind half a second of device work fill the queue; while the caller waits for room, another Python thread
    goes on ticking."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2511_15369_b200 import api
    c = api.gelu_prepare(2.5e-4, 16, 8.2 / 255, -123)
    x = torch.arange(-32, 32, dtype=torch.int32, device="cuda")
    out = api.gelu(x, c)
    torch.cuda.synchronize()
    stop, gaps = threading.Event(), []

    def tick():
        last = time.perf_counter()
        while not stop.is_set():
            time.sleep(0.002)
            now = time.perf_counter()
            gaps.append(now - last)
            last = now
    t = threading.Thread(target=tick)
    t.start()
    time.sleep(0.05)
    began = time.perf_counter()
    torch.cuda._sleep(1_000_000_000)                           # half a second at 1.9 GHz
    for _ in range(6000):
        api.gelu(x, c, out=out)
    enqueued = time.perf_counter() - began
    stop.set()
    t.join()
    torch.cuda.synchronize()
    assert enqueued > 0.25, "the queue never filled up (%.3f s): this shows nothing" % enqueued
    assert max(gaps) < 0.1, max(gaps)

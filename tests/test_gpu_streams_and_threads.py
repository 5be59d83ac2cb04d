"""A cache used from several streams and threads: what a call leaves behind is complete on every stream, and a call that waits for
the GPU does not stop the other threads of the program."""
import threading
import time

import torch
import pytest

import paper_2502_02617_b200 as pq
from paper_2502_02617_b200 import synthetic

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def test_a_launch_that_blocks_does_not_hold_the_interpreter_lock():
    cache = pq.PolarQuantCache(1, 4, 1, 128, capacity=64, device=DEV)
    K, V = synthetic.kv_like(1, 64, 1, 128, torch.bfloat16, DEV)
    cache.encode(K, V, torch.tensor([0, 64], dtype=torch.int32, device=DEV))
    q = synthetic.queries(2, 1, 4, 128, torch.bfloat16, DEV)
    out = cache.attend(q)
    torch.cuda.synchronize()
    ticks, stop = [time.perf_counter()], threading.Event()

    def tick():
        while not stop.is_set():
            time.sleep(0.002)
            ticks.append(time.perf_counter())

    thread = threading.Thread(target=tick)
    thread.start()
    torch.cuda._sleep(1_500_000_000)          # three quarters of a second of the GPU: the launches below fill its queue
    t0 = time.perf_counter()
    for _ in range(3000):
        cache.attend(q, out=out)
    blocked = time.perf_counter() - t0
    stop.set()
    thread.join()
    torch.cuda.synchronize()
    assert blocked > 0.4                      # the queue was full
    assert max(b - a for a, b in zip(ticks, ticks[1:])) < 0.2

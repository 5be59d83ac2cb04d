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


def _codebooks():
    """Level 1 shifted: not the analytic codebook."""
    cen, bnd = pq.pq_fit_codebooks()
    cen, bnd = cen.clone(), bnd.clone()
    cen[:16] += 0.1
    bnd[:15] += 0.1
    return cen, bnd


@pytest.mark.parametrize("n", [20, 300])
def test_new_codebooks_are_complete_on_every_stream(n):
    cache, want = pq.PolarQuantCache(1, 2, 2, 128, capacity=n, device=DEV), pq.PolarQuantCache(1, 2, 2, 128, n, device=DEV, codebooks=_codebooks())
    K, V = synthetic.kv_like(3, n, 2, 128, torch.bfloat16, DEV)
    cu, side = torch.tensor([0, n], dtype=torch.int32, device=DEV), torch.cuda.Stream()
    want.encode(K, V, cu)
    torch.cuda.synchronize()
    torch.cuda._sleep(400_000_000)            # the current stream is busy
    cache.set_codebooks(*_codebooks())
    cache.encode(K, V, cu, stream=side)
    torch.cuda.synchronize()
    assert torch.equal(cache.unpack(n)[0], want.unpack(n)[0])


def test_codebooks_fitted_on_one_stream_serve_another():
    n = 300
    cache, want = (pq.PolarQuantCache(1, 2, 2, 128, capacity=n, device=DEV) for _ in range(2))
    K, V = synthetic.kv_like(4, n, 2, 128, torch.bfloat16, DEV)
    cu, side = torch.tensor([0, n], dtype=torch.int32, device=DEV), torch.cuda.Stream()
    hist = want.fit_online_codebooks(K, V)
    want.encode(K, V, cu)
    torch.cuda.synchronize()
    assert torch.equal(cache.fit_online_codebooks(K, V, stream=side), hist)
    cache.encode(K, V, cu)
    assert torch.equal(cache.centroids, want.centroids) and torch.equal(cache.unpack(n)[0], want.unpack(n)[0])


def test_chunks_on_several_streams_do_not_share_scratch():
    n, n_q = 4000, 64
    cache = pq.PolarQuantCache(2, 16, 4, 128, capacity=n, device=DEV)
    K, V = synthetic.kv_like(5, 2 * n, 4, 128, torch.bfloat16, DEV)
    cache.encode(K, V, torch.tensor([0, n, 2 * n], dtype=torch.int32, device=DEV))
    qs = [synthetic.queries(6 + i, 2 * n_q, 16, 128, torch.bfloat16, DEV).view(2, n_q, 16, 128) for i in range(10)]
    want = [cache.attend_multi(q) for q in qs]
    streams = [torch.cuda.Stream() for _ in qs]              # more than workspaces are kept for
    outs = [torch.empty_like(q) for q in qs]
    torch.cuda.synchronize()
    for _ in range(5):
        for q, out, s in zip(qs, outs, streams):
            cache.attend_multi(q, out=out, stream=s)
        torch.cuda.synchronize()
        assert all(torch.equal(o, w) for o, w in zip(outs, want))


def test_arguments_that_the_entry_points_take_and_refuse():
    cache = pq.PolarQuantCache(2, 4, 2, 128, capacity=64, device=DEV)
    K, V = synthetic.kv_like(7, 20, 2, 128, torch.bfloat16, DEV)
    cache.encode(K, V, torch.tensor([0, 10, 20], dtype=torch.int32, device=DEV))
    q = synthetic.queries(8, 2, 4, 128, torch.bfloat16, DEV)
    with pytest.raises((AssertionError, AttributeError)):    # the log-sum-exp has nowhere to go
        pq.pq_decode_attention_lse(cache.S, cache.tables, q, cache.cache, cache.lens, 2, 64, 64, 0.1, torch.empty_like(q), None,
                                   cache.workspace, cache.status)
    general = pq.GeneralPolarQuantCache(2, 4, 2, 64, (3, 3), 64, device=DEV)
    Kg, Vg = synthetic.kv_like(9, 20, 2, 64, torch.float32, DEV)
    general.encode(Kg, Vg, torch.tensor([0, 10, 20], dtype=torch.int32, device=DEV))
    qg = synthetic.queries(10, 2, 4, 64, torch.float32, DEV)
    flat = torch.empty(2 * 4 * 64, device=DEV)               # an output of another shape
    assert torch.equal(general.attend(qg, out=flat).view(2, 4, 64), general.attend(qg))

"""Attention captured in a CUDA graph and replayed on changed inputs: a replay repeats the call's number (the persistent
head_dim-128 kernel tags its scratch with it) and must still wait for every part."""
import pytest
import torch

import paper_2502_02617_b200 as pq
from paper_2502_02617_b200 import synthetic

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("d,B,Hq,Hkv,n", [(128, 2, 8, 2, 9000), (128, 1, 16, 2, 20000), (128, 2, 4, 2, 300), (64, 2, 8, 2, 700)])
def test_replayed_attention_equals_eager_calls(d, B, Hq, Hkv, n):
    cache = pq.PolarQuantCache(B, Hq, Hkv, d, capacity=n + 8, seed=3, device=DEV)
    K, V = synthetic.kv_like(1, B * n, Hkv, d, torch.bfloat16, DEV)
    cache.encode(K, V, torch.arange(0, B + 1, dtype=torch.int32, device=DEV) * n)
    q = synthetic.queries(2, B, Hq, d, torch.bfloat16, DEV)
    k1, v1 = synthetic.kv_like(3, B, Hkv, d, torch.bfloat16, DEV)
    out = torch.empty_like(q)
    start = cache.lens.clone()
    cache.attend(q, out=out)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        cache.append(k1, v1)
        cache.attend(q, out=out)
    for step in range(4):
        q.copy_(synthetic.queries(10 + step, B, Hq, d, torch.bfloat16, DEV))
        k1.copy_(synthetic.kv_like(20 + step, B, Hkv, d, torch.bfloat16, DEV)[0])
        graph.replay()
        got = out.clone()
        assert cache.lens.cpu().tolist() == [n + 1 + step] * B
        assert torch.equal(got, cache.attend(q))       # same kernel, same split, same order of additions
    cache.lens.copy_(start)
    cache.check_status()

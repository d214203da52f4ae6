"""The calls under stream capture: a captured sequence replayed on new inputs gives the bits of the
calls issued directly. Covers the dependent, cooperative and cluster launches of every route."""

import pytest
import torch

import paper_2609_31568_gb300 as pkg
from paper_2609_31568_gb300 import scale as S

pytestmark = pytest.mark.gpu

BASE = dict(num_q_heads=8, num_kv_heads=2, sub_chunk=256, n_tokens=4096, max_cluster_subchunks=4, n_sink=64,
            n_local=256)


@pytest.fixture(scope="session", autouse=True)
def _built():
    pkg.build()
    S.load()


def _random(n, heads, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(n, heads, 128, generator=gen, device="cuda", dtype=torch.bfloat16)


@pytest.mark.parametrize("mode", [S.SCALE_MODE_PER_CLUSTER, S.SCALE_MODE_PER_SUBCHUNK])
@pytest.mark.parametrize("over", [dict(block_size=64, top_k=8), dict(block_size=64, top_k=8, theta=0.5),
                                  dict(block_size=1, top_k=300), dict(block_size=64, top_k=8, n_tokens=8192)])
def test_captured_layer_equals_direct_calls(mode, over):
    p = S.params(**{**BASE, **over})
    n = p.n_tokens
    q, k, v = (torch.empty(n, h, 128, dtype=torch.bfloat16, device="cuda") for h in (8, 2, 2))
    buf, ref = pkg.allocate(p, mode), pkg.allocate(p, mode)
    for t in (q, k, v):
        t.copy_(_random(n, t.shape[1], 1))
    pkg.run_path(p, mode, q, k, v, ref)  # first use outside the capture
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        pkg.run_path(p, mode, q, k, v, buf)
    for seed in (2, 3):
        for i, t in enumerate((q, k, v)):
            t.copy_(_random(n, t.shape[1], 10 * seed + i))
        graph.replay()
        pkg.run_path(p, mode, q, k, v, ref)
        torch.cuda.synchronize()
        assert torch.equal(buf.out, ref.out)
        assert S.scale_get_device_status(buf.ws) == S.SCALE_OK


@pytest.mark.parametrize("heads", [(8, 2), (7, 1)])
def test_captured_decode_equals_direct_calls(heads):
    hq, hkv = heads
    n, steps = 4096, 4
    p = S.params(**{**BASE, "num_q_heads": hq, "num_kv_heads": hkv}, block_size=1, top_k=100, theta=0.9)
    k, v = _random(n, hkv, 1), _random(n, hkv, 2)
    q = torch.empty(steps, hq, 128, dtype=torch.bfloat16, device="cuda")
    outs = [torch.empty(steps, hq, 128, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    cache = [torch.empty(S.scale_decode_cache_size(p), dtype=torch.uint8, device="cuda") for _ in range(2)]
    ws = [torch.empty(S.scale_decode_workspace_size(p), dtype=torch.uint8, device="cuda") for _ in range(2)]
    for x in range(2):
        S.scale_workspace_init(ws[x])

    def run(x):
        S.scale_decode_cache_init(cache[x])
        for i in range(steps):
            S.scale_decode_step(p, n - steps + i, q[i], k, v, cache[x], outs[x][i], ws[x])

    q.copy_(_random(steps, hq, 3))
    run(1)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        run(0)
    for seed in (4, 5):
        base = _random(1, hq, seed).float()
        q.copy_(base + 0.2 * _random(steps, hq, 10 * seed).float())
        graph.replay()
        run(1)
        torch.cuda.synchronize()
        assert torch.equal(outs[0], outs[1])
        assert S.scale_get_device_status(ws[0]) == S.SCALE_OK

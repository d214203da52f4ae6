"""A value row that is not finite reaches no output row whose 128-row query block ends before it: an
output row attends to keys at or before itself, and the kernel's key tiles end with the query block."""

import pytest
import torch

import paper_2609_31568_gb300 as pkg
from paper_2609_31568_gb300 import scale as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="session", autouse=True)
def _built():
    pkg.build()
    S.load()


@pytest.mark.parametrize("hq,hkv,n,sub", [
    (28, 4, 8192, 512),    # odd group: the last head's CTAs take two query blocks
    (28, 4, 8190, 512),    # a ragged second block
    (3, 1, 16384, 384),    # three blocks per sub-chunk: pairs and a single one
    (5, 1, 8192, 512),     # every tile on an SM of its own
    (8, 2, 8192, 512),     # even group
])
@pytest.mark.parametrize("block,topk", [(64, 8), (1, 300)])
def test_future_value_rows_stay_out(hq, hkv, n, sub, block, topk):
    gen = torch.Generator(device="cuda").manual_seed(n + hq)
    q, k, v = (torch.randn(n, h, 128, generator=gen, device="cuda", dtype=torch.bfloat16) for h in (hq, hkv, hkv))
    mode = S.SCALE_MODE_PER_SUBCHUNK
    p = S.params(num_q_heads=hq, num_kv_heads=hkv, sub_chunk=sub, n_tokens=n, max_cluster_subchunks=1,
                 block_size=block, top_k=topk, n_sink=128, n_local=sub)
    buf = pkg.allocate(p, mode)
    pkg.run_path(p, mode, q, k, v, buf)
    clean = buf.out.clone()
    for row in (n - 1, n - 130, n // sub * sub - 1, n // 2 // sub * sub + 129):
        bad = v.clone()
        bad[row] = float("inf")
        S.scale_sparse_prefill(p, mode, 0, n, q, k, bad, buf.unit_start, buf.n_units, buf.sel_blocks, buf.sel_count,
                               buf.out, buf.ws)
        start = row // sub * sub
        first = start + (row - start) // 128 * 128  # first row of the query block that holds `row`
        assert torch.equal(buf.out[:first], clean[:first]), row
    assert S.scale_get_device_status(buf.ws) == S.SCALE_OK

"""A unit's block-level scores and blocks are the same, bit for bit, whichever calls its sequence is cut
into: one over the whole sequence, some units each, one unit each. On both sides of the line between
the kernels, and at every cluster size of the one-launch kernel."""

import pytest
import torch

import paper_2609_31568_gb300 as pkg
from paper_2609_31568_gb300 import scale as S

pytestmark = pytest.mark.gpu

# (query heads, KV heads, blocks, block, sub-chunks, cluster cap, threshold)
CASES = [
    (4, 1, 64, 64, 16, 4, -1.0),
    (32, 8, 250, 128, 32, 8, 0.5),     # 32 units: clusters of 4 CTAs; one unit: 16
    (32, 8, 513, 32, 80, 1, -1.0),     # 80 units: one CTA a unit
    (28, 4, 301, 17, 40, 5, -1.0),     # ragged everything
    (3, 1, 700, 7, 155, 3, 0.3),       # more units than SMs
    (8, 8, 1024, 8, 64, 8, -1.0),
    (32, 8, 1024, 32, 64, 4, -1.0),    # the last sequence of the one-launch kernel ...
    (32, 8, 1025, 32, 64, 4, -1.0),    # ... and the first of the others
    (10, 1, 300, 16, 30, 1, -1.0),     # a group of 10: the others
    (16, 4, 5000, 4, 20, 2, -1.0),     # more than 4096 blocks
]


@pytest.fixture(scope="session", autouse=True)
def _built():
    pkg.build()
    S.load()


@pytest.mark.parametrize("mode", [S.SCALE_MODE_PER_CLUSTER, S.SCALE_MODE_PER_SUBCHUNK])
@pytest.mark.parametrize("hq,hkv,nb,block,m,cap,theta", CASES)
def test_scores_do_not_depend_on_the_call(hq, hkv, nb, block, m, cap, theta, mode):
    n = nb * block
    sub = -(-n // m)
    p = S.params(num_q_heads=hq, num_kv_heads=hkv, sub_chunk=sub, n_tokens=n, max_cluster_subchunks=cap,
                 block_size=block, top_k=min(20, nb // 4), n_sink=block, n_local=sub // 2, theta=theta)
    gen = torch.Generator(device="cuda").manual_seed(nb)
    m = -(-n // sub)
    q = torch.randn(n, hq, 128, generator=gen, device="cuda", dtype=torch.bfloat16)
    q += torch.randn(m, hq, 128, generator=gen, device="cuda").to(torch.bfloat16).repeat_interleave(sub, 0)[:n]
    k = torch.randn(n, hkv, 128, generator=gen, device="cuda", dtype=torch.bfloat16)
    step = sub * (cap if mode == S.SCALE_MODE_PER_CLUSTER else 1)
    whole = None
    for per_call in (m, 16, 5, 1):  # units (outer chunks) per call
        buf = pkg.allocate(p, mode, want_scores=True)
        S.scale_build_reps(p, q, k, buf.reps, buf.fingerprints, buf.unit_start, buf.n_units, buf.ws)
        for t in range(0, n, per_call * step):
            S.scale_select(p, mode, t, min(n, t + per_call * step), buf.reps, buf.fingerprints, buf.unit_start,
                           buf.n_units, buf.sel_blocks, buf.sel_count, buf.sel_scores, buf.ws)
        torch.cuda.synchronize()
        assert S.scale_get_device_status(buf.ws) == S.SCALE_OK
        u = int(buf.n_units) if mode == S.SCALE_MODE_PER_CLUSTER else m
        got = (buf.sel_scores[:u].view(torch.int32), buf.sel_blocks[:u], buf.sel_count[:u])
        if whole is None:
            whole = got
        for a, b in zip(got, whole):
            assert torch.equal(a, b), per_call

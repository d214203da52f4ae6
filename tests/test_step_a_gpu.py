"""Step (a) at the sizes where its tiles end: clusters of many outer chunks, chunks longer than shared
memory, clusters of more sub-chunks than a warp has lanes; representatives of blocks that share a CTA.

Clusters: the queries of a sub-chunk are one coordinate direction, so every cosine is exactly 0 or 1 and the
table is known. Representatives: a mean of B bf16 values in fp32, at most B + 32 additions and a division,
each off by 2^-24 of a sum of at most sum |k|.
"""

import pytest
import torch

import paper_2609_31568_gb300 as pkg
from paper_2609_31568_gb300 import scale as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="session", autouse=True)
def _built():
    pkg.build()
    S.load()


def _clusters(topic, per_outer, cap):
    starts = []
    for c in range(0, len(topic), per_outer):
        end = min(len(topic), c + per_outer)
        a = c
        while a < end:
            starts.append(a)
            j = a + 1
            while j < end and j - a < cap and topic[j] == topic[a]:
                j += 1
            a = j
    return starts


@pytest.mark.parametrize("m,per_outer,cap,stay", [
    (1, 1, 3, 0.5),
    (5, 4, 2, 0.5),
    (300, 16, 16, 0.9),
    (2000, 40, 40, 0.99),    # a cluster takes two rounds of a warp
    (700, 600, 9, 0.8),      # 5,400 cosines of a chunk: two windows of 455 sub-chunks
    (900, 900, 5000, 0.9),   # an anchor's cosines do not fit shared memory
    (130, 64, 64, 0.97),     # 4,096: the most that shared memory keeps
    (8200, 8, 8, 0.7),       # 1,025 chunks
    (3000, 3, 2, 0.0),       # every sub-chunk a cluster
    (3000, 3000, 3000, 1.0),  # and one cluster of all
])
@pytest.mark.parametrize("calls", [1, 4])  # over the whole sequence, or appended by range
def test_clusters_of_known_cosines(m, per_outer, cap, stay, calls):
    sub = 2
    n = m * sub - 1
    gen = torch.Generator().manual_seed(m)
    jump = (torch.rand(m, generator=gen) >= stay).long()
    topic = (jump * torch.randint(1, 100, (m,), generator=gen)).cumsum(0) % 100
    q = torch.zeros(n, 1, 128, dtype=torch.bfloat16, device="cuda")
    rows = torch.arange(n, device="cuda")
    q[rows, 0, topic.cuda()[rows // sub]] = 2.0
    k = torch.zeros(n, 1, 128, dtype=torch.bfloat16, device="cuda")
    p = S.params(num_q_heads=1, num_kv_heads=1, sub_chunk=sub, n_tokens=n, max_cluster_subchunks=cap,
                 outer_chunk=per_outer * sub, theta=0.5, block_size=64, top_k=1, n_sink=0, n_local=0)
    buf = pkg.allocate(p, S.SCALE_MODE_PER_CLUSTER)
    buf.unit_start.fill_(-5)
    step = -(-m // (calls * per_outer)) * per_outer * sub
    for t in range(0, n, step):
        S.scale_build_reps_range(p, t, min(n, t + step), q, k, buf.reps, buf.fingerprints, buf.unit_start,
                                 buf.n_units, buf.ws)
    want = _clusters(topic.tolist(), per_outer, cap)
    assert int(buf.n_units) == len(want)
    assert buf.unit_start.tolist() == want + [m] * (m + 1 - len(want))


@pytest.mark.parametrize("hkv", [1, 2, 3, 5, 8, 12, 33, 64])
@pytest.mark.parametrize("n,block,paged", [(1, 64, False), (700, 1, False), (701, 7, False), (999, 8, False),
                                           (1000, 15, False), (4097, 16, False), (4001, 64, False), (4001, 64, True),
                                           (5000, 100, False), (9000, 4096, False)])
def test_representatives(hkv, n, block, paged):
    gen = torch.Generator(device="cuda").manual_seed(n + hkv)
    k = torch.randn(n, hkv, 128, generator=gen, device="cuda", dtype=torch.bfloat16)
    q = torch.zeros(n, hkv, 128, dtype=torch.bfloat16, device="cuda")
    p = S.params(num_q_heads=hkv, num_kv_heads=hkv, sub_chunk=64, n_tokens=n, max_cluster_subchunks=4, block_size=block,
                 top_k=1, n_sink=0, n_local=64)
    nb = -(-n // block)
    buf = pkg.allocate(p, S.SCALE_MODE_PER_CLUSTER)
    reps = torch.full((hkv, nb, 128), float("nan"), device="cuda")
    if paged:
        pages = -(-n // 64)
        table = torch.randperm(pages + 2, generator=gen, device="cuda")[:pages]
        pool = torch.full((pages + 2, 64, hkv, 128), float("nan"), dtype=torch.bfloat16, device="cuda")
        full = torch.zeros(pages * 64, hkv, 128, dtype=torch.bfloat16, device="cuda")
        full[:n] = k
        pool[table] = full.view(pages, 64, hkv, 128)
        kv = S.kv_pages(pool, pool, table.int(), 64)
        S.scale_build_reps_paged(p, q, kv, reps, buf.fingerprints, buf.unit_start, buf.n_units, buf.ws)
    else:
        S.scale_build_reps(p, q, k, reps, buf.fingerprints, buf.unit_start, buf.n_units, buf.ws)
    for b in range(nb):
        rows = k[b * block: (b + 1) * block].double()
        bound = (len(rows) + 33) * 2.0 ** -24 * rows.abs().mean(0)
        assert torch.all((reps[:, b].double() - rows.mean(0)).abs() <= bound)

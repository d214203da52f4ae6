"""Token-level selection of few units (one read of K, planes of logits, vote and top-k in one launch)
at the sizes where its tiles, slices and digits end: against the same rule in 64 bits.

Scores: the dot products are exact in the three bf16 parts up to fp32 accumulation, so a logit of size
|z| is off by a few 2^-24 |z|, which the exponential turns into the same relative error of the score:
2e-5 holds for |z| up to about 60. A selection may differ only by tokens whose score is that close to
the k-th one; equal keys give bit-equal scores, so exact ties have to go to the lower token: of the tokens
with equal keys that a selection cuts, it holds the first ones, also across the slices of the CTAs (some
two hundred tokens with 19 CTAs a unit, a few thousand in the longest).

The planes live in the space of the packed keys; where they do not fit, K is read twice by other kernels.
"""

import math

import pytest
import torch

import paper_2609_31568_gb300 as pkg
from paper_2609_31568_gb300 import scale as S

pytestmark = pytest.mark.gpu

PER_SUB = S.SCALE_MODE_PER_SUBCHUNK

# (query heads, KV heads, tokens, sub-chunk, sinks, window, k, repeated keys)
CASES = [
    (4, 1, 700, 100, 0, 0, 1, False),
    (4, 1, 701, 100, 3, 50, 8, False),        # odd rows: padded planes; a sink inside the first quad
    (4, 1, 2048, 128, 64, 128, 64, False),    # 16 units: four column tiles
    (8, 2, 4099, 512, 130, 100, 64, True),    # exact ties across slices
    (7, 1, 5003, 1000, 130, 64, 4999, False),  # k >= candidates
    (5, 1, 6001, 1500, 127, 1, 300, True),
    (3, 3, 4000, 1000, 129, 256, 2047, False),
    (16, 16, 3000, 1000, 128, 64, 0, False),  # nothing selected
    (1, 1, 40000, 20000, 128, 512, 19000, True),
    (32, 8, 30011, 2048, 128, 1024, 2000, False),
    # keys larger than L2 keeps: the unit tiles side by side, the last of two units and of one
    (32, 8, 50001, 2048, 128, 1024, 2000, False),
    (28, 4, 100003, 8192, 130, 128, 5500, True),
    # slices longer than the keys that stay in shared memory
    (1, 1, 400_000, 25_000, 0, 0, 4000, False),
    (1, 1, 400_000, 25_000, 0, 0, 4000, True),
]
TWO_READS = [  # planes that do not fit
    (16, 16, 3000, 1000, 0, 64, 0, False),    # nothing selected
    (28, 4, 100003, 8192, 130, 128, 300, True),
    (1, 1, 10_400_003, 5_200_064, 128, 0, 30000, False),
]


def _planes_fit(hq, hkv, n, sub, sink, k):
    """Whether a call of the last 16 units at most has room for their planes of logits."""
    m, slots = -(-n // sub), -(-(sink + k) // 128) * 128
    units = min(m, 16)
    scratch = -(-units * (3 * 2048 + 16 + 2 * 256) * 4 // 256) * 256
    return scratch + units * hq * (-(-n // 4) * 4) * 4 <= 2 * m * hkv * slots * 256


@pytest.fixture(scope="session", autouse=True)
def _built():
    pkg.build()
    S.load()


@pytest.mark.parametrize("hq,hkv,n,sub,sink,local,k,ties", CASES + TWO_READS)
def test_few_unit_token_selection(hq, hkv, n, sub, sink, local, k, ties):
    assert _planes_fit(hq, hkv, n, sub, sink, k) == ((hq, hkv, n, sub, sink, local, k, ties) in CASES)
    g = hq // hkv
    gen = torch.Generator(device="cuda").manual_seed(n)
    keys = torch.randn(n, hkv, 128, generator=gen, device="cuda", dtype=torch.bfloat16)
    if ties:
        keys = keys[:97].repeat(-(-n // 97), 1, 1)[:n].contiguous()
    p = S.params(num_q_heads=hq, num_kv_heads=hkv, sub_chunk=sub, n_tokens=n, max_cluster_subchunks=1,
                 block_size=1, top_k=k, n_sink=sink, n_local=local)
    buf = pkg.allocate(p, PER_SUB, want_scores=True)
    m = -(-n // sub)
    fp = 0.3 * torch.randn(m, hq * 128, generator=gen, device="cuda")
    first = max(0, m - 16)
    cut = False  # a selection held some of a group of equal keys
    for scores in (buf.sel_scores, None):  # with and without the scores asked for
        buf.sel_blocks.fill_(-7)
        S.scale_select_tokens(p, PER_SUB, first * sub, n, keys, fp, None, None, buf.sel_blocks, buf.sel_count,
                              scores, buf.ws)
        torch.cuda.synchronize()
        assert S.scale_get_device_status(buf.ws) == S.SCALE_OK
        for u in range(first, m):
            w = max(0, u * sub - local)
            cand = max(0, w - sink)
            got = buf.sel_blocks[u, : max(k, 1)].long()
            count = int(buf.sel_count[u])
            assert count == min(k, cand)
            if scores is not None:
                off = torch.ones(n, dtype=torch.bool, device="cuda")
                off[sink:max(w, sink)] = False
                assert torch.equal(torch.isnan(scores[u]), off)
            if cand == 0 or k == 0:
                continue
            z = torch.einsum("jgd,tjd->jgt", fp[u].view(hkv, g, 128).double(), keys[sink:w].double())
            ref = torch.softmax(z, dim=-1).sum((0, 1))
            if scores is not None:
                torch.testing.assert_close(scores[u, sink:w].double(), ref, rtol=2e-5, atol=1e-10)
            want = torch.sort(torch.sort(ref, descending=True, stable=True)[1][:k])[0] + sink
            assert torch.all(got[count:] == -1) if count < k else True
            assert torch.all(got[1:count] > got[: count - 1]) and got[0] >= sink and got[count - 1] < w
            assert torch.equal(got[:count], want) or _near(got[:count], want, ref, sink, 2e-5)
            if ties and cand > k:  # of the equal keys, those at the same place of each 97, the first ones
                for r in range(97):
                    group = torch.arange(sink + (r - sink) % 97, w, 97, device="cuda")
                    mine = got[:count][got[:count] % 97 == r]
                    assert torch.equal(mine, group[: len(mine)])
                    cut |= 0 < len(mine) < len(group)
    assert cut or not ties


@pytest.mark.parametrize("n,spread", [(16384, 2.0), (100003, 2.0), (100003, 3.0), (100003, 8.0)])
def test_error_of_spread_logits(n, spread):
    """Exact logits (a coordinate of a bf16 key each): what is left of a score's error is the exponential's,
    two ulps at most and less than one in the root mean square, and the rounding of its argument, a
    difference of at most a few units for the tokens that carry the score: 2^-24 8 ln 2 / sqrt(3) for the
    largest of them. 1e-7 together, 1.6e-7 with a margin; with the product of logit and scale rounded
    before the difference and references between which the factors are approximate 1.7e-7 to 3.2e-7."""
    sub = 1024
    m = -(-n // sub)
    rel = []
    for seed in range(8):
        gen = torch.Generator(device="cuda").manual_seed(seed)
        keys = torch.zeros(n, 1, 128, dtype=torch.bfloat16, device="cuda")
        keys[:, 0, :8] = spread * torch.randn(n, 8, generator=gen, device="cuda")
        fp = torch.eye(8, 128, device="cuda").flatten().repeat(m, 1)
        p = S.params(num_q_heads=8, num_kv_heads=1, sub_chunk=sub, n_tokens=n, max_cluster_subchunks=1,
                     block_size=1, top_k=2048, n_sink=0, n_local=0)
        buf = pkg.allocate(p, PER_SUB, want_scores=True)
        S.scale_select_tokens(p, PER_SUB, (m - 4) * sub, n, keys, fp, None, None, buf.sel_blocks, buf.sel_count,
                              buf.sel_scores, buf.ws)
        torch.cuda.synchronize()
        for u in range(m - 4, m):
            ref = torch.softmax(keys[: u * sub, 0, :8].double(), 0).sum(1)
            rel.append(float((buf.sel_scores[u, : u * sub].double() - ref).norm() / ref.norm()))
    mean = sum(rel) / len(rel)
    assert mean < 1.6e-7, mean


@pytest.mark.parametrize("scale", [1e3, 1e9, 1e15, 1e30])
def test_one_token_far_above_the_others(scale):
    """A logit whose own rounding is larger than the range of the exponential: its token has the whole
    probability of every head, in a tile of candidates and in the last, partial one."""
    n, sub, topk = 3000, 1000, 300
    assert _planes_fit(4, 1, n, sub, 0, topk)
    gen = torch.Generator(device="cuda").manual_seed(5)
    keys = torch.randn(n, 1, 128, generator=gen, device="cuda", dtype=torch.bfloat16)
    keys[:, 0, 0] = 0.0
    keys[700, 0, 0], keys[1990, 0, 0] = scale, -scale
    fp = 0.1 * torch.randn(3, 4, 128, generator=gen, device="cuda")
    fp[:, :, 0] = 0.77
    p = S.params(num_q_heads=4, num_kv_heads=1, sub_chunk=sub, n_tokens=n, max_cluster_subchunks=1, block_size=1,
                 top_k=topk, n_sink=0, n_local=0)
    buf = pkg.allocate(p, PER_SUB, want_scores=True)
    S.scale_select_tokens(p, PER_SUB, 0, n, keys, fp.flatten(1), None, None, buf.sel_blocks, buf.sel_count,
                          buf.sel_scores, buf.ws)
    for u in (1, 2):
        scores = buf.sel_scores[u, : u * sub]
        assert torch.all(torch.isfinite(scores)) and 3.99 < float(scores[700]) < 4.01
        assert float(scores.sum() - scores[700]) < 1e-3 and 700 in buf.sel_blocks[u].tolist()


def _near(got, want, ref, sink, rel):
    """Whether every token in only one of the lists scores within `rel` of the k-th score."""
    kth = ref[want - sink].min()
    one = torch.cat([got[~torch.isin(got, want)], want[~torch.isin(want, got)]])
    return bool(torch.all((ref[one - sink] / kth).log().abs() < 2 * rel)) and math.isfinite(float(kth))

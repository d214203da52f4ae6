"""Block-level selection against the same rule in 64 bits, at the sizes where the one-launch kernel's
runs, groups and clusters end and on both sides of the line to the kernels for sequences of more work.

Scores: the error of a logit is the relative error of the score. The tensor-core kernel adds 48 partial
products per logit into an fp32 accumulator, each addition off by at most 2^-23 (truncation) of a partial
sum, taken as at most the largest logit: 48 * 2^-23 * max|z|. The one-launch kernel's fp32 sums of 128
products in trees stay far below that. A selection may differ only by blocks whose score is that close to
the k-th one; equal representatives give bit-equal scores, so exact ties have to go to the lower block.
"""

import pytest
import torch

import paper_2609_31568_gb300 as pkg
from paper_2609_31568_gb300 import scale as S

pytestmark = pytest.mark.gpu

PER_SUB = S.SCALE_MODE_PER_SUBCHUNK

# (query heads, KV heads, tokens, sub-chunk, block, sinks, window, k, units of the call, repeated rows)
CASES = [
    (4, 1, 1100, 64, 8, 0, 0, 1, 16, False),
    (4, 1, 1100, 64, 8, 0, 0, 1, 18, False),        # clusters of 4 CTAs
    (1, 1, 4000, 1000, 3, 5, 17, 100, 4, True),     # ragged blocks, exact ties across the ranks
    (2, 1, 4000, 1000, 16, 16, 100, 249, 4, False),  # k = candidates - 1 and candidates for some units
    (3, 1, 5000, 500, 7, 40, 100, 33, 9, False),
    (5, 1, 5000, 500, 7, 40, 100, 33, 10, True),
    (12, 2, 5000, 1000, 9, 0, 1, 64, 5, False),
    (28, 4, 8200, 1024, 33, 64, 128, 20, 9, False),
    (64, 8, 8200, 1024, 64, 64, 128, 20, 8, True),
    (256, 64, 3000, 1000, 64, 64, 128, 8, 3, False),  # the most heads of the one-launch kernel
    (260, 52, 3000, 1000, 64, 64, 128, 8, 3, False),  # and beyond
    (10, 1, 3000, 1000, 32, 0, 0, 8, 3, False),       # group of 10: the other kernels
    (4, 1, 40000, 10000, 10, 0, 0, 4000, 4, False),   # 4000 blocks
    (32, 8, 70000, 10000, 16, 64, 128, 1000, 7, True),  # more than 4096 blocks
    (4, 2, 3000, 1000, 64, 64, 128, 0, 3, False),     # nothing selected
    (4, 1, 300000, 10000, 64, 64, 1024, 64, 30, True),  # many units, 4,688 blocks
    (32, 8, 16416, 1000, 32, 0, 0, 64, 7, True),     # the most units of clusters of 16
    (32, 8, 16416, 1000, 32, 0, 0, 64, 8, True),     # and one unit more: clusters of 8
    (32, 8, 16384, 1024, 32, 0, 0, 64, 14, False),   # the most units of those
    (32, 8, 16384, 1024, 32, 0, 0, 64, 15, False),
    # the kernels for sequences of more work: 16-byte and 4-byte loads, segments of several unit tiles
    (32, 8, 66000, 500, 64, 64, 128, 20, 9, True),     # 1,032 blocks
    (28, 4, 66000, 300, 61, 40, 100, 33, 15, False),   # 1,082 blocks
    (8, 8, 66000, 220, 64, 0, 1, 64, 300, True),
    (256, 64, 6400, 64, 64, 64, 128, 8, 4, False),
    (10, 1, 40000, 10000, 9, 0, 0, 300, 4, True),      # more than 4096 blocks
]


@pytest.fixture(scope="session", autouse=True)
def _built():
    pkg.build()
    S.load()


@pytest.mark.parametrize("hq,hkv,n,sub,block,sink,local,k,units,ties", CASES)
def test_block_selection_of_units(hq, hkv, n, sub, block, sink, local, k, units, ties):
    g, m, nb = hq // hkv, -(-n // sub), -(-n // block)
    gen = torch.Generator(device="cuda").manual_seed(n + hq)
    reps = torch.randn(hkv, nb, 128, generator=gen, device="cuda")
    if ties:
        reps = reps[:, :61].repeat(1, -(-nb // 61), 1)[:, :nb].contiguous()
    fp = 0.3 * torch.randn(m, hq * 128, generator=gen, device="cuda")
    p = S.params(num_q_heads=hq, num_kv_heads=hkv, sub_chunk=sub, n_tokens=n, max_cluster_subchunks=1,
                 block_size=block, top_k=k, n_sink=sink, n_local=local)
    buf = pkg.allocate(p, PER_SUB, want_scores=True)
    first = max(0, m - units)
    for scores in (buf.sel_scores, None):  # with and without the scores asked for
        buf.sel_blocks.fill_(-7)
        S.scale_select(p, PER_SUB, first * sub, n, reps, fp, None, None, buf.sel_blocks, buf.sel_count, scores, buf.ws)
        torch.cuda.synchronize()
        assert S.scale_get_device_status(buf.ws) == S.SCALE_OK
        for u in range(first, m):
            lo = sink // block
            hi = max(lo, -(-max(0, u * sub - local) // block))
            count = int(buf.sel_count[u])
            assert count == min(k, hi - lo)
            if scores is not None:
                off = torch.ones(nb, dtype=torch.bool, device="cuda")
                off[lo:hi] = False
                assert torch.equal(torch.isnan(scores[u]), off)
            if hi == lo or k == 0:
                continue
            z = torch.einsum("jgd,jbd->jgb", fp[u].view(hkv, g, 128).double(), reps[:, lo:hi].double())
            ref = torch.softmax(z, dim=-1).sum((0, 1))
            tol = 48 * 2.0 ** -23 * max(1.0, float(z.abs().max()))
            if scores is not None:
                torch.testing.assert_close(scores[u, lo:hi].double(), ref, rtol=tol, atol=1e-10)
            got = buf.sel_blocks[u, :k].long()
            want = torch.sort(torch.sort(ref, descending=True, stable=True)[1][:k])[0] + lo
            assert torch.all(got[count:] == -1)
            got = got[:count]
            assert torch.all(got[1:] > got[:-1]) and got[0] >= lo and got[-1] < hi
            if not torch.equal(got, want):
                kth = ref[want - lo].min()
                one = torch.cat([got[~torch.isin(got, want)], want[~torch.isin(want, got)]])
                assert torch.all((ref[one - lo] / kth).log().abs() < 2 * tol)
                if ties:  # of a tied group that is cut, the lower blocks
                    for r in torch.unique((one - lo) % 61):
                        mine = got[(got - lo) % 61 == r]
                        assert torch.equal(mine, torch.arange(len(mine), device="cuda") * 61 + r + lo)


@pytest.mark.parametrize("nb,batch", [(2064, 1024), (2062, 256)])  # 16-byte and 4-byte loads
def test_large_terms_are_summed_against_their_maximum(nb, batch):
    """A head whose probability lies on 32 equal blocks, met by the lanes of a warp after blocks 6 to 8 below
    them (by lane 0 before): the large terms of its sum are exactly 1, as in a sum over the known maximum.
    What is left in the root mean square over 64 gaps is the rounding of a lane's sum (2^-24 / sqrt(3)), the
    reciprocal (an ulp: 2^-23 / sqrt(3)) and the additions over the lanes, of nearly equal values and so
    nearly exact: 8e-8, and half as much again for them (measured 4e-8). Terms taken against a reference 6
    to 8 below them carry the rounding of an argument of 8 to 12 log2 units as well: 1.6e-7."""
    lane = torch.arange(32, device="cuda") * (4 if nb % 4 == 0 else 1)
    block, sub = 2, 8
    n = nb * block
    m = -(-n // sub)
    reps = torch.zeros(1, nb, 128, device="cuda")
    reps[0, :, 1] = -200.0
    low, high = lane.clone(), lane + batch
    low[0], high[0] = batch, 0
    reps[0, low, :2] = 0.0
    reps[0, high, 0], reps[0, high, 1] = 7.875, 0.0
    fp = torch.zeros(m, 128, device="cuda")
    fp[:, 0] = 0.75 + (torch.arange(m, device="cuda") % 64 + 1) / 256  # the gap / 7.875; exact logits
    fp[:, 1] = 1.0
    p = S.params(num_q_heads=1, num_kv_heads=1, sub_chunk=sub, n_tokens=n, max_cluster_subchunks=1, block_size=block,
                 top_k=8, n_sink=0, n_local=0)
    buf = pkg.allocate(p, PER_SUB, want_scores=True)
    S.scale_select(p, PER_SUB, 0, n, reps, fp, None, None, buf.sel_blocks, buf.sel_count, buf.sel_scores, buf.ws)
    torch.cuda.synchronize()
    rel = []
    for u in range(m - 64, m):
        z = fp[u, 0].double() * reps[0, : u * sub // block, 0].double() + reps[0, : u * sub // block, 1].double()
        ref = torch.softmax(z, 0)[high]
        rel.append(((buf.sel_scores[u][high].double() - ref) / ref).mean())
    rms = float(torch.stack(rel).square().mean().sqrt())
    assert rms < 1.2e-7, rms

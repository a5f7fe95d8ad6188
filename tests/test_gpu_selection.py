"""The selection where its form changes: few candidates (all ranked directly), one more, and cut-offs decided by age."""
import pytest
import torch

from oracle.kvc_oracle import KVCOracle
from paper_2604_16734_b200.binding import KVC_SCORE_KEYDIFF, Kvc
from parity_util import compare_chunk
from test_gpu_attention_shapes import launch_shape

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,B,chunks", [
    (torch.float32, 96, (96, 32, 64, 65, 1)),           # 96, 128 (ranked directly), 129 and 96 candidates
    (torch.bfloat16, 40, (40, 33, 1, 2)),               # windows of one and two rows
])
def test_candidate_counts(dtype, B, chunks):
    torch.manual_seed(B)
    d, hq, hkv = 64, 2, 2
    kvc = Kvc(1, hq, hkv, d, dtype, B, max(chunks))
    orc = KVCOracle(1, hq, hkv, d, B, 32)
    pos = 0
    for n in chunks:
        q, k, v = (torch.randn(n, h, d).to(dtype) for h in (hq, hkv, hkv))
        compare_chunk(kvc, orc, 0, q, k, v, pos)        # retained sets bit-exact above a gap of 1e-3
        pos += n


@pytest.mark.parametrize("groups", [1, 3])
@pytest.mark.parametrize("B,n", [(64, 64), (600, 400)])
def test_equal_scores_keep_the_oldest(groups, B, n):
    # keys of a group are identical, so their scores are equal: whole groups stay by score, the cut-off group by age
    d, w, N = 64, 32, 4 * n - 7
    gen = torch.Generator().manual_seed(groups)
    u = torch.nn.functional.normalize(torch.randn(d, generator=gen), dim=0)
    rank = torch.arange(N) % groups                                   # group 0 scores highest
    k = ((3.0 * (1.0 - rank.float() / groups))[:, None] * u)[:, None, :].contiguous()
    v = torch.randn(N, 1, d, generator=gen)
    q = (u * 8.0).expand(N, 1, d).contiguous()
    kvc = Kvc(1, 1, 1, d, torch.float32, B, n)
    held = []
    for p in range(0, N, n):
        m = min(n, N - p)
        kvc.prefill_chunk(0, q[p:p + m].cuda(), k[p:p + m].cuda(), v[p:p + m].cuda(), p)
        cand, new = held + list(range(p, p + m - w)), list(range(p + m - w, p + m))
        if len(cand) + w > B:
            cand = sorted(cand, key=lambda t: (int(rank[t]), t))[:B - w]
        held = sorted(cand + new)
    assert kvc.status() == 0
    _, _, pos, length = kvc.cache_view(0)
    assert length == B and pos[0, :B].sort().values.cpu().tolist() == held


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_equal_keys_at_the_cutoff(dtype):
    # a caller that gives two blocks the same positions: entries with equal score and position, two of them at ranks 15 and
    # 16 of the 16 that stay
    d, w, B, n = 64, 4, 20, 16
    torch.manual_seed(2)
    k = torch.randn(1, 1, d, device="cuda").expand(n, 1, d).to(dtype).contiguous()
    q = torch.randn(1, 1, d, device="cuda").expand(n, 1, d).to(dtype).contiguous()
    kvc = Kvc(1, 1, 1, d, dtype, B, n, w)
    vs = [torch.randn(n, 1, d, device="cuda").to(dtype) for _ in range(2)]
    for v in vs:
        kvc.prefill_chunk(0, q, k, v, 0)
    assert kvc.status() == 0
    _, V, pos, length = kvc.cache_view(0)
    held = pos[0, :B].cpu().tolist()
    assert length == B and sorted(held) == sorted(2 * list(range(8)) + [12, 13, 14, 15])
    rows = {tuple(x[0].tolist()) for v in vs for x in v.cpu()}
    assert all(tuple(x) in rows for x in V[0, :B].cpu().tolist())
    assert len({tuple(x) for x in V[0, :B].cpu().tolist()}) == B


@pytest.mark.parametrize("dtype,d,n,B", [
    (torch.float32, 64, 16, 21),                        # ranked directly, one of two equal keys stays
    (torch.float32, 64, 100, 150),                      # the keys of the cut-off bin ranked; equal keys end at the cut-off
    (torch.bfloat16, 128, 100, 151),                    # ... or lie across it
    (torch.float32, 128, 200, 300),                     # decided bit by bit
    (torch.bfloat16, 64, 200, 301),
    (torch.bfloat16, 64, 3200, 5001),                   # keys re-read from the workspace, move lists in global memory
])
def test_equal_keys_across_the_cutoff(dtype, d, n, B):
    # two blocks with the same positions behind one far ahead of them, all scores equal: exactly B - w candidates stay, the
    # oldest first, and the last block's window with them
    w, starts = 4, (1 << 20, 0, 0)
    torch.manual_seed(n)
    k = torch.randn(1, 1, d, device="cuda").expand(n, 1, d).to(dtype).contiguous()
    q = torch.randn(1, 1, d, device="cuda").expand(n, 1, d).to(dtype).contiguous()
    vs = [torch.randn(n, 1, d, device="cuda").to(dtype) for _ in starts]
    kvc = Kvc(1, 1, 1, d, dtype, B, n, w)
    held = []
    for p, v in zip(starts, vs):
        kvc.prefill_chunk(0, q, k, v, p)
        cand, new = held + list(range(p, p + n - w)), list(range(p + n - w, p + n))
        held = (sorted(cand)[:B - w] if len(cand) + w > B else cand) + new
    assert kvc.status() == 0
    _, V, pos, length = kvc.cache_view(0)
    pos = pos[0, :B].cpu().tolist()
    assert length == B and sorted(pos) == sorted(held)
    where = {tuple(row): (b, p + i) for b, (p, v) in enumerate(zip(starts, vs)) for i, row in enumerate(v[:, 0].cpu().tolist())}
    rows = [where[tuple(row)] for row in V[0, :B].cpu().tolist()]
    assert [p for _, p in rows] == pos and len(set(rows)) == B
    assert all((2, n - w + i) in rows for i in range(w))


@pytest.mark.parametrize("hq,hkv,d,dtype,n,B,form", [
    (16, 4, 64, torch.bfloat16, 333, 1500, "beside"),   # the compress kernel runs beside the attention
    (4, 4, 128, torch.bfloat16, 65, 90, "ranked"),      # candidates ranked directly
    (2, 1, 64, torch.bfloat16, 2300, 7000, "global"),   # keys re-read from the workspace, move lists in global memory
    (4, 1, 64, torch.float32, 64, 128, "cuda cores"),
])
def test_query_agnostic_selection_ahead_of_the_attention(hq, hkv, d, dtype, n, B, form):
    # calls enqueued back to back, so that a selection runs while its block's attention does, against plain stream order
    # (flag 8), bit for bit: everything that is compared is copied or selected, and the sums are taken in the same order.
    # The outputs would show a move that overwrites a row the attention still reads.
    layers, blocks, w = 2, B // n + 4, 32
    n_cand = B + n - w
    torch.manual_seed(n)
    qkv = [[torch.randn(blocks * n, h, d, device="cuda").to(dtype) for h in (hq, hkv, hkv)] for _ in range(layers)]
    held = []
    for flags in (8, 0, 0, 0, 0):
        kvc = Kvc(layers, hq, hkv, d, dtype, B, n, w, flags=flags, policy=KVC_SCORE_KEYDIFF)
        if form == "beside":                             # (the rule: all CTAs of both kernels fit the GPU)
            row_tiles, split, pairs = launch_shape(kvc, n, B)
            tiles = -(-n // (128 // (hq // hkv)))
            assert hkv * (tiles * split if row_tiles == 1 else tiles - pairs) + hkv * min(16, 148 // hkv, -(-n_cand // 256)) <= 148
        assert (n_cand <= 128) == (form == "ranked") and (n_cand > 6144 and n > 2048) == (form == "global")
        outs = [kvc.prefill_chunk(l, *(x[p:p + n] for x in qkv[l]), p) for p in range(0, blocks * n, n) for l in range(layers)]
        assert kvc.status() == 0
        held.append(outs + [t[:, :B].clone() for l in range(layers) for t in kvc.cache_view(l)[:3]])
    for got in held[1:]:
        assert all(torch.equal(a, b) for a, b in zip(held[0], got))


@pytest.mark.parametrize("dtype,d,n,B", [(torch.bfloat16, 64, 30, 50), (torch.float32, 128, 30, 50), (torch.bfloat16, 128, 300, 500),
                                         (torch.float32, 64, 300, 500)])
def test_query_agnostic_ties_between_cached_and_new_entries(dtype, d, n, B):
    # all keys equal, so age alone decides, and the last block's positions lie between those of the blocks before it: the
    # cut-off falls inside it, with cached entries (positions read from the cache) and new ones (computed) on either side
    hq = hkv = 2
    w, starts = 4, (1000, 2000, 1500)
    torch.manual_seed(d)
    k = torch.randn(1, hkv, d, device="cuda").expand(n, hkv, d).to(dtype).contiguous()
    kvc = Kvc(1, hq, hkv, d, dtype, B, n, w, policy=KVC_SCORE_KEYDIFF)
    held = []
    for p in starts:
        q, v = (torch.randn(n, h, d, device="cuda").to(dtype) for h in (hq, hkv))
        kvc.prefill_chunk(0, q, k, v, p)
        cand, new = held + list(range(p, p + n - w)), list(range(p + n - w, p + n))
        kept = sorted(cand)[:B - w] if len(cand) + w > B else cand
        dropped, held = set(cand) - set(kept), kept + new
    assert {x // 500 for x in kept} == {2, 3} and {x // 500 for x in dropped} == {3, 4}
    assert kvc.status() == 0
    _, _, pos, length = kvc.cache_view(0)
    assert length == B and all(sorted(row) == sorted(held) for row in pos[:, :B].cpu().tolist())

"""The launch shapes of the tensor-core attention and their edges: two row tiles per CTA with an odd last one, one row tile
with one to many key tiles, key splits over clusters of 2, 4 and 8 CTAs (some without a key tile of the first rows), group
sizes that leave rows of a tile unused."""
import ctypes

import pytest
import torch

from oracle.kvc_oracle import KVCOracle
from paper_2604_16734_b200.binding import KVC_FLAG_ASYNC_COMPRESS, Kvc
from parity_util import compare_chunk

pytestmark = pytest.mark.gpu


def launch_shape(kvc, n, n_c):
    x = [ctypes.c_int() for _ in range(3)]
    assert kvc._lib.kvc_attention_shape(kvc._h, n, n_c, 1, *(ctypes.byref(v) for v in x)) == 0
    return tuple(v.value for v in x)


@pytest.mark.parametrize("hq,hkv,d,B,chunks,shape", [
    (1, 1, 64, 40, (1, 40, 9), (1, 1, 0)),                # one row; one key tile, then two
    (32, 32, 128, 140, (140, 129, 128), (1, 1, 0)),       # two row tiles per kv-head, the second with 12 rows / one row
    (28, 4, 128, 260, (260, 577), (1, 1, 0)),             # G = 7: 126 rows per tile; 577 tokens
    (4, 1, 128, 2000, (2000, 40, 33), (1, 8, 0)),         # clusters of 8
    (4, 2, 64, 2500, (2500, 40, 1), (1, 8, 0)),           # the same with d = 64
    (4, 1, 128, 1100, (1100, 40, 33), (1, 4, 0)),         # clusters of 4
    (8, 2, 64, 700, (700, 256, 255), (1, 4, 0)),
    (32, 8, 128, 900, (900, 196, 197), (1, 2, 0)),        # clusters of 2
    (16, 16, 128, 130, (130, 1200), (2, 1, 5)),           # two row tiles per CTA
    (16, 16, 128, 130, (130, 1660), (2, 1, 6)),           # two row tiles per CTA, odd count: the last CTA has one
    (12, 4, 64, 140, (140, 1100), (1, 1, 0)),             # G = 3, long block after a short cache
    (28, 4, 128, 150, (150, 784, 703), (2, 1, 7)),        # pairs first, then single row tiles (the last one ragged)
    (32, 8, 64, 300, (300, 600, 641), (2, 1, 7)),         # the same with d = 64; more single tiles than pairs
    (16, 16, 64, 1400, (1400, 154, 33), (1, 4, 0)),       # compress clusters of six, where seven would not all fit the GPU
    (24, 24, 64, 1300, (1300, 60), (1, 4, 0)),            # five for six
])
def test_launch_shapes(hq, hkv, d, B, chunks, shape):
    torch.manual_seed(B + hq)
    kvc = Kvc(1, hq, hkv, d, torch.bfloat16, B, max(chunks))
    orc = KVCOracle(1, hq, hkv, d, B, 32)
    pos = 0
    for n in chunks:
        last = launch_shape(kvc, n, min(pos, B))
        q, k, v = (torch.randn(n, h, d).to(torch.bfloat16) for h in (hq, hkv, hkv))
        compare_chunk(kvc, orc, 0, q, k, v, pos)        # output within 2e-2 (or one bf16 ulp of the rounded oracle value)
        pos += n
    assert last == shape                                # (row tiles per CTA, key split, pairs) of the last block


@pytest.mark.parametrize("hq,hkv,d,B,chunks,window,flags", [
    (28, 4, 128, 300, (300, 130, 129), 32, 0),        # 224 observer rows, two to four key tiles
    (32, 8, 64, 200, (200, 90, 33), 64, 0),           # 256 observer rows, the most that are scored in the fused kernel
    (20, 4, 64, 260, (260, 60, 27), 26, 0),           # 130 observer rows, the fewest that take the wide form
    (66, 2, 64, 200, (200, 64, 31), 8, 0),            # 264: a score kernel of its own
    (64, 8, 128, 300, (300, 64, 64), 32, KVC_FLAG_ASYNC_COMPRESS),   # side stream without room for two launches
    (28, 4, 64, 150, (150, 784, 784), 32, KVC_FLAG_ASYNC_COMPRESS),  # pairs and single row tiles, SMs left for compress
])
def test_observer_rows(hq, hkv, d, B, chunks, window, flags):
    torch.manual_seed(B + hq)
    kvc = Kvc(1, hq, hkv, d, torch.bfloat16, B, max(chunks), window, flags=flags)
    orc = KVCOracle(1, hq, hkv, d, B, window)
    pos = 0
    for n in chunks:
        q, k, v = (torch.randn(n, h, d).to(torch.bfloat16) for h in (hq, hkv, hkv))
        compare_chunk(kvc, orc, 0, q, k, v, pos)
        pos += n


def test_output_at_sixteen_byte_alignment():
    # `out` needs 16-byte alignment only: at 16 modulo 32 the one-row-tile launch stores in smaller pieces, same values
    n, hq, hkv, d = 70, 8, 2, 128
    torch.manual_seed(1)
    q, k, v = (torch.randn(n, h, d, device="cuda", dtype=torch.bfloat16) for h in (hq, hkv, hkv))
    a, b = Kvc(1, hq, hkv, d, torch.bfloat16, 100, n), Kvc(1, hq, hkv, d, torch.bfloat16, 100, n)
    whole = torch.zeros(n * hq * d + 24, device="cuda", dtype=torch.bfloat16)
    shifted = whole[8:8 + n * hq * d].view(n, hq, d)
    assert shifted.data_ptr() % 32 == 16
    ref = a.prefill_chunk(0, q, k, v, 0)
    b.prefill_chunk(0, q, k, v, 0, shifted)
    assert a.status() == 0 and b.status() == 0
    assert torch.equal(ref, shifted) and not whole[:8].any() and not whole[8 + n * hq * d:].any()


@pytest.mark.parametrize("hq,hkv,d,n,B,window", [
    (28, 4, 128, 784, 2048, 32),                      # pairs and single row tiles
    (32, 8, 64, 640, 1000, 32),
    (32, 32, 128, 700, 500, 8),                       # the first block already evicts
    (28, 4, 128, 576, 1024, 32),                      # 224 / 256 observer rows: a score kernel of its own on the side
    (64, 8, 128, 64, 300, 32),                        # stream, where two fused launches would not fit beside the attention
])
def test_compress_on_a_side_stream_gives_the_same_bits(hq, hkv, d, n, B, window):
    layers, N = 2, (B // n + 4) * n
    torch.manual_seed(n)
    qkv = [[torch.randn(N, h, d, device="cuda", dtype=torch.bfloat16) for h in (hq, hkv, hkv)] for _ in range(layers)]
    res = []
    for flags in (0, KVC_FLAG_ASYNC_COMPRESS):
        kvc = Kvc(layers, hq, hkv, d, torch.bfloat16, B, n, window, flags=flags)
        outs = [kvc.prefill_chunk(l, *(x[p:p + n] for x in qkv[l]), p) for p in range(0, N, n) for l in range(layers)]
        kvc.join()
        assert kvc.status() == 0
        res.append((outs, [t for l in range(layers) for t in kvc.cache_view(l)[:3]],
                    kvc.workspace_view(kvc.slot_of(layers - 1))[1][:, :B + n - window].clone()))
    (outs_a, cache_a, score_a), (outs_b, cache_b, score_b) = res
    assert all(torch.equal(a, b) for a, b in zip(outs_a, outs_b))
    assert all(torch.equal(a[:, :B], b[:, :B]) for a, b in zip(cache_a, cache_b))
    assert torch.equal(score_a, score_b)


@pytest.mark.parametrize("hq,hkv,d,n,blocks,row_tiles", [
    (4, 2, 128, 128, 9, 1),                           # one to nine key tiles: below, at and around a ring of three per kind,
    (4, 2, 64, 100, 9, 1),                            # the appended tile in each of its slots
    (32, 32, 64, 640, 3, 2),                          # two row tiles per CTA: a ring of two, blocks of five tiles
    (28, 4, 128, 784, 2, 2),                          # pairs and single row tiles on the same ring
])
def test_key_tiles_around_the_ring(hq, hkv, d, n, blocks, row_tiles):
    torch.manual_seed(n)
    kvc = Kvc(1, hq, hkv, d, torch.bfloat16, n * blocks, n, flags=4)     # KVC_FLAG_NO_KEY_SPLIT
    orc = KVCOracle(1, hq, hkv, d, n * blocks, 32)
    for i in range(blocks):
        q, k, v = (torch.randn(n, h, d).to(torch.bfloat16) for h in (hq, hkv, hkv))
        compare_chunk(kvc, orc, 0, q, k, v, i * n)    # (and the cached rows, bit for bit)
    assert launch_shape(kvc, n, n * (blocks - 1))[0] == row_tiles


@pytest.mark.parametrize("hq,hkv,d", [(2, 2, 64), (6, 2, 128)])
@pytest.mark.parametrize("n_c", [1, 31, 32, 33, 64, 95, 96, 97, 127, 129])
def test_mask_at_the_quarters_of_a_tile(hq, hkv, d, n_c):
    # the last cache tile ends at row n_c, the block's own tile at every row's token: limits around multiples of 32 columns
    torch.manual_seed(n_c)
    kvc = Kvc(1, hq, hkv, d, torch.bfloat16, n_c, 130, 1)
    orc = KVCOracle(1, hq, hkv, d, n_c, 1)
    for pos, n in ((0, n_c), (n_c, 130)):
        q, k, v = (torch.randn(n, h, d).to(torch.bfloat16) for h in (hq, hkv, hkv))
        compare_chunk(kvc, orc, 0, q, k, v, pos)

"""The CUDA-core attention and score kernels at the edges of their tiles: every row tile (8, 16, 32 rows), key splits over
clusters of 1 to 8 CTAs, 16 and 32 keys per score CTA, more than 128 observer rows, both head dimensions, remainders of one."""
import pytest
import torch

from oracle.kvc_oracle import KVCOracle
from paper_2604_16734_b200.binding import KVC_FLAG_CUDA_CORES, Kvc
from parity_util import compare_chunk

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,hq,hkv,d,B,chunks", [
    (torch.float32, 1, 1, 64, 40, (1, 40, 9, 17)),                 # one row, one key; a single step
    (torch.float32, 4, 1, 128, 1200, (1200, 33, 32, 1)),           # few rows, many keys: cluster of 8
    (torch.float32, 8, 8, 128, 300, (300, 64, 65, 31)),            # cluster of 2 / 4
    (torch.float32, 7, 1, 64, 100, (100, 130, 129)),               # 224 observer rows (two groups), G no power of two
    (torch.float32, 16, 4, 128, 260, (260, 196, 197)),             # 32 rows per CTA
    (torch.float32, 8, 2, 128, 530, (530, 300, 271)),              # 16 rows per CTA, several waves
    (torch.float32, 16, 16, 64, 400, (400, 100, 51)),              # 32 keys per score CTA
    (torch.bfloat16, 4, 2, 128, 150, (150, 33, 90)),               # bf16 through the same kernels (diagnostic flag)
])
def test_tile_edges(dtype, hq, hkv, d, B, chunks):
    torch.manual_seed(B + d)
    kvc = Kvc(1, hq, hkv, d, dtype, B, max(chunks), flags=KVC_FLAG_CUDA_CORES if dtype == torch.bfloat16 else 0)
    orc = KVCOracle(1, hq, hkv, d, B, 32)
    pos = 0
    for n in chunks:
        q, k, v = (torch.randn(n, h, d).to(dtype) for h in (hq, hkv, hkv))
        compare_chunk(kvc, orc, 0, q, k, v, pos)        # tolerances of the parity contract: 1e-4 (fp32), 2e-2 (bf16)
        pos += n

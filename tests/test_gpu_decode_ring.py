"""Decode attention over 16-bit rows: row counts around the tiles (16 rows), a CTA's steps (64 or 128) and the ring of three
tiles per warp, with few heads (eight warps to a CTA, clusters) and with many (four warps, no cluster); an output that is
only as aligned as a float."""
import math

import pytest
import torch

import paper_2406_02069_b200 as pkv
from helpers import packed_rows

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("dtype,d", [("bf16", 128), ("fp16", 64)])
@pytest.mark.parametrize("heads,lens", [
    (3, [16, 17, 130, 385]), (2, [383, 384, 1153]), (1, [3071, 3073]),
    (80, [15, 63, 64, 65]), (80, [191, 192, 193, 257]), (40, [448, 449, 1, 575, 2, 127, 129, 400]),
], ids=lambda v: str(v[0]) if isinstance(v, list) else str(v))
def test_counts_around_the_tiles(heads, lens, dtype, d):
    group = 3
    cfg = pkv.make_config(num_layers=1, num_q_heads=group * heads, num_kv_heads=heads, head_dim=d, window=1, pool_kernel=1,
                          dtype=dtype, avg_budget=1)
    t = {"bf16": torch.bfloat16, "fp16": torch.float16}[dtype]
    lens = [n + 1 for n in lens]                             # a window of one row; a budget beyond every length keeps all
    kl = max(lens)
    counts = [pkv.kept_count(cfg, kl, n) for n in lens]
    g = torch.Generator().manual_seed(41)
    rows = pkv.total_rows(cfg, kl, lens)
    k, v = (torch.randn(rows, d, generator=g).to(t) for _ in range(2))
    q = (2.0 * torch.randn(len(lens), group * heads, d, generator=g)).to(t)
    whole = torch.full((len(lens) * group * heads * d + 1,), 7.0, device=DEV)
    out = whole[1:].view(len(lens), group * heads, d)
    pkv.decode_attention(cfg, q.to(DEV), k.to(DEV), v.to(DEV), lens, kl, out)
    got = out.cpu().double()
    for b, h, sl in packed_rows(counts, heads):
        x = q[b, h * group:(h + 1) * group].double() @ k[sl].double().T / math.sqrt(d)
        w = torch.softmax(x, 1)
        # fp32 logits (sum |q k| at most 256 here, 2^-22 of it) and weights, products of 24-bit weights summed in fp32
        bound = 2e-4 * (w @ v[sl].double().abs()) + 1e-6
        assert torch.all((got[b, h * group:(h + 1) * group] - w @ v[sl].double()).abs() <= bound), (b, h)
    assert whole[0].item() == 7.0

"""Decode attention over the compact cache at the edges of its split: query heads per KV head around the blocks (of four
with 16-bit rows, of up to eight in fp32), head sizes, types, and row counts around a step, a cluster's slices and a single
row."""
import numpy as np
import pytest
import torch

import oracle
import paper_2406_02069_b200 as pkv
from helpers import packed_rows

pytestmark = pytest.mark.gpu
DEV = "cuda"


# (query heads per KV head, KV heads, head size, dtype, window, k_layer, lengths)
CASES = [
    (1, 2, 128, "bf16", 1, 0, [2, 9]),               # one row a head
    (1, 3, 64, "fp16", 3, 60, [64, 67, 900]),        # 63 rows: just below a step
    (2, 2, 128, "fp16", 4, 60, [500]),               # 64 rows
    (3, 2, 128, "bf16", 5, 60, [500]),               # 65 rows, a group padded to four heads
    (4, 2, 64, "fp32", 8, 505, [2000, 700]),
    (4, 8, 128, "bf16", 32, 3900, [5000]),           # long lists over clusters of eight
    (7, 1, 128, "bf16", 8, 1017, [1500]),            # 1025 rows over eight CTAs of one head, two blocks of query heads
    (8, 2, 64, "bf16", 8, 200, [300, 5000, 301]),
    (12, 1, 128, "fp16", 8, 120, [4000]),            # three blocks of query heads
    (5, 2, 128, "bf16", 8, 120, [4000, 90]),         # two, one head in the second
    (6, 1, 64, "fp16", 8, 700, [4000]),              # ... two heads
    (12, 2, 128, "fp32", 8, 120, [4000, 90]),        # fp32: a block of eight and half a one
    (8, 40, 128, "fp32", 2, 30, [100, 101, 102, 103]),   # enough heads that no cluster forms
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "g%d_h%d_d%d_%s_k%d" % (c[0], c[1], c[2], c[3], c[4] + c[5]))
def test_decode_against_the_oracle(case):
    group, heads, d, dtype, window, kl, lens = case
    cfg = pkv.make_config(num_layers=1, num_q_heads=group * heads, num_kv_heads=heads, head_dim=d, window=window, pool_kernel=1,
                          dtype=dtype, avg_budget=window)
    t = {"fp32": torch.float32, "bf16": torch.bfloat16, "fp16": torch.float16}[dtype]
    g = torch.Generator().manual_seed(13)
    rows = pkv.total_rows(cfg, kl, lens)
    k, v = (torch.randn(rows, d, generator=g).to(t) for _ in range(2))
    q = (2.0 * torch.randn(len(lens), group * heads, d, generator=g)).to(t)
    out = torch.full((len(lens), group * heads, d), 7.0, device=DEV)
    pkv.decode_attention(cfg, q.to(DEV), k.to(DEV), v.to(DEV), lens, kl, out)
    # the same rows through pages of odd size give the same bits
    page = 7
    counts = [pkv.kept_count(cfg, kl, n) for n in lens]
    pages = [pkv.pages_needed(cfg, kl, n, page) for n in lens]
    total = heads * sum(pages)
    table = torch.randperm(total, generator=g).to(torch.int32)
    k_pool, v_pool = (torch.zeros(total, page, d, dtype=t) for _ in range(2))
    at = 0
    for b, h, sl in packed_rows(counts, heads):
        tab = table[at: at + pages[b]].numpy()
        oracle.scatter_paged(k[sl], tab, page, k_pool)
        oracle.scatter_paged(v[sl], tab, page, v_pool)
        at += pages[b]
    ws = pkv.new_workspace(cfg, len(lens), max(lens), DEV)
    paged = torch.zeros_like(out)
    pkv.decode_attention_paged(cfg, q.to(DEV), table.to(DEV), k_pool.to(DEV), v_pool.to(DEV), lens, kl, paged, ws)
    pkv.check_status(ws)
    assert torch.equal(out, paged)
    got = out.cpu().numpy()
    for b, h, sl in packed_rows(counts, heads):
        for j in range(group):
            hq = h * group + j
            want = oracle.decode_attention(q[b, hq], k[sl], v[sl])
            # exponents x = q.k log2(e)/sqrt(d): at most d / 8 + 5 roundings of terms whose absolute sum is below 64 here
            # move x by less than 64 * 21 * 2^-24 = 8e-5 and a weight by the factor 2^8e-5; sums of the weights add less
            # than 1e-5: 7e-5 of the output over |V|
            bound = oracle.decode_attention(q[b, hq], k[sl], v[sl].abs())
            assert np.all(np.abs(got[b, hq] - want) <= 7e-5 * bound + 1e-7), (b, hq)


@pytest.mark.parametrize("what", ["inf", "-inf", "both signs", "nan", "small weight", "last row"])
@pytest.mark.parametrize("dtype,d,group", [("fp32", 128, 4), ("bf16", 128, 4), ("fp16", 128, 5), ("bf16", 64, 1), ("fp16", 64, 2)])
def test_infinities_and_nan_in_the_values_stay_in_their_channel(dtype, d, group, what):
    heads, window, kl, lens = 2, 4, 296, [700, 90]
    cfg = pkv.make_config(num_layers=1, num_q_heads=group * heads, num_kv_heads=heads, head_dim=d, window=window, pool_kernel=1,
                          dtype=dtype, avg_budget=window)
    t = {"fp32": torch.float32, "bf16": torch.bfloat16, "fp16": torch.float16}[dtype]
    g = torch.Generator().manual_seed(17)
    rows = pkv.total_rows(cfg, kl, lens)
    k, v = (torch.randn(rows, d, generator=g).to(t) for _ in range(2))
    q = (1.5 * torch.randn(len(lens), group * heads, d, generator=g)).to(t)
    inf = float("inf")
    if what == "both signs":
        v[10, 3], v[200, 3], v[10, 40] = inf, -inf, -inf
    elif what == "small weight":                             # another row's logit some 40 binades above
        v[10, 3] = inf
        k[20] = (q[0, 0].float() * (40.0 / 1.4427 * d ** 0.5 / q[0, 0].float().square().sum())).to(t)
    elif what == "last row":
        v[rows - 1, d - 1], v[299, 0] = -inf, inf
    else:
        v[10, 3] = float(what)
    out = torch.zeros(len(lens), group * heads, d, device=DEV)
    pkv.decode_attention(cfg, q.to(DEV), k.to(DEV), v.to(DEV), lens, kl, out)
    counts, got = [pkv.kept_count(cfg, kl, n) for n in lens], out.cpu().double()
    for b, h, sl in packed_rows(counts, heads):
        for j in range(group):
            hq = h * group + j
            w = torch.softmax(k[sl].double() @ q[b, hq].double() / d ** 0.5, 0)[:, None]
            want = (w * v[sl].double()).sum(0)
            assert torch.equal(torch.isnan(got[b, hq]), torch.isnan(want)), (b, hq)
            special = ~torch.isfinite(want)
            assert torch.equal(got[b, hq][special & ~torch.isnan(want)], want[special & ~torch.isnan(want)]), (b, hq)
            bound = (w * v[sl].double().abs()).sum(0)        # as in the test above
            assert torch.all((got[b, hq] - want).abs()[~special] <= 7e-5 * bound[~special] + 1e-7), (b, hq)

"""Pooling, selection and placement at the edges of the selection kernel: prefix lengths around its instances (2048,
4096, 8192 and 16384 positions a CTA) and cluster sizes, budgets from one row to all but one, ties, clustered winners,
pool widths on both sides of the register path, score rows off the 16-byte grid.  Lists are compared exactly."""
import numpy as np
import pytest
import torch

import oracle
import paper_2406_02069_b200 as pkv

pytestmark = pytest.mark.gpu
DEV = "cuda"
ALPHA = 4


def scores_of(kind, heads, P, seed):
    g = torch.Generator().manual_seed(seed)
    if kind == "normal":
        return torch.rand(heads, P, generator=g) ** 8
    if kind == "ties":                                       # few distinct values: plateaus far longer than the budget
        return torch.randint(0, 3, (heads, P), generator=g).float()
    if kind == "equal":
        return torch.full((heads, P), 0.25)
    if kind == "tiny":                                       # scales off the kernel's absolute bins, and rows within one bin
        return (torch.rand(heads, P, generator=g) ** 8) * 1e-12
    if kind == "negative":
        return torch.rand(heads, P, generator=g) - 2
    if kind == "huge":
        return (torch.rand(heads, P, generator=g) ** 8) * 1e6
    if kind == "flat":
        return (1 + 0.02 * torch.rand(heads, P, generator=g)) / P
    s = torch.rand(heads, P, generator=g) * 1e-6             # "crowd": the winners sit in one stretch, with one huge score
    at = (P * 5) // 7
    s[:, at: at + P // 16 + 2] += 1.0 + torch.rand(heads, min(P // 16 + 2, P - at), generator=g)
    s[:, 1] = 3.0e4
    return s


# (prefix length, k, pool width, mean pool, scores, leading dimension minus prefix length)
CASES = [
    (1, 1, 3, 0, "normal", 3), (2, 1, 1, 0, "normal", 0), (31, 30, 5, 0, "normal", 1), (33, 5, 7, 1, "normal", 3),
    (255, 254, 7, 0, "ties", 0), (2048, 100, 7, 0, "normal", 0), (2049, 100, 5, 0, "normal", 3), (2047, 700, 7, 1, "ties", 1),
    (4095, 1, 7, 0, "crowd", 1), (4096, 96, 7, 0, "equal", 0), (4097, 4096, 9, 0, "normal", 7), (8191, 188, 7, 0, "normal", 1),
    (8192, 3000, 5, 0, "crowd", 0), (8193, 600, 7, 0, "normal", 3), (8200, 8000, 11, 1, "normal", 0), (20000, 1023, 7, 0, "crowd", 0),
    (20001, 1024, 7, 0, "crowd", 3), (32736, 3900, 7, 0, "normal", 0), (40000, 20000, 5, 0, "ties", 0), (65537, 188, 33, 0, "normal", 7),
    (131072, 188, 7, 0, "normal", 0), (131072, 9000, 3, 1, "normal", 0), (131071, 64, 7, 0, "equal", 1), (131073, 64, 7, 0, "crowd", 3),
    (3000, 200, 35, 0, "normal", 0),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "P%d_k%d_w%d_%s_%s" % (c[0], c[1], c[2], "avg" if c[3] else "max", c[4]))
def test_selection_is_exact(case):
    check_selection(case, 0)


# slices of 4097 .. 8192 positions by half-size CTAs, where the configuration caps the sweeps' CTAs
@pytest.mark.parametrize("case", [c for c in CASES if c[0] in (4096, 4097, 8191, 8192, 8193, 20001, 32736, 40000)],
                         ids=lambda c: "P%d_k%d_%s" % (c[0], c[1], c[4]))
def test_selection_beside_other_layers_is_exact(case):
    check_selection(case, 74)


def check_selection(case, sweep_ctas):
    P, k, w, avg, kind, slack = case
    heads, d = 2, 64
    short = max(1, P // 3)                                   # a second, shorter sequence in the same launch
    lens = [P + ALPHA, short + ALPHA]
    cfg = pkv.make_config(num_layers=1, num_q_heads=heads, num_kv_heads=heads, head_dim=d, window=ALPHA, pool_kernel=w, dtype="bf16",
                          avg_budget=ALPHA, pool_kind=avg, sweep_ctas=sweep_ctas)
    s = torch.zeros(2, heads, P + slack)
    s[0, :, :P] = scores_of(kind, heads, P, 3)
    s[1, :, :short] = scores_of(kind, heads, short, 4)
    ws = pkv.new_workspace(cfg, 2, max(lens), DEV)
    idx = torch.full((pkv.total_rows(cfg, k, lens),), -1, dtype=torch.int32, device=DEV)
    pkv.select_topk(cfg, s.to(DEV), lens, k, idx, ws)
    pkv.check_status(ws)
    got, at = idx.cpu().numpy(), 0
    pool = oracle.pool_avg if avg else oracle.pool_max
    for b, n in enumerate(lens):
        prefix = n - ALPHA
        for h in range(heads):
            want = oracle.select_topk(pool(s[b, h, :prefix].numpy(), w), min(k, prefix))
            want = np.concatenate([want, np.arange(prefix, n)])
            assert np.array_equal(got[at: at + len(want)], want), (b, h)
            at += len(want)


SCALES = ["tiny", "negative", "huge", "flat"]


# one CTA, two, eight; bounds per CTA and for the cluster; more rows than runs; all but a few
@pytest.mark.parametrize("kind", SCALES)
@pytest.mark.parametrize("P,k,w,avg", [(1500, 40, 1, 0), (4000, 96, 7, 0), (8190, 3000, 3, 0), (12000, 480, 7, 1), (20000, 1100, 5, 0),
                                       (33000, 3000, 1, 0), (100000, 64, 21, 0), (131040, 96, 7, 0), (131001, 5000, 1, 0), (131072, 130000, 3, 1)])
def test_selection_is_exact_on_any_scale(P, k, w, avg, kind):
    check_selection((P, k, w, avg, kind, 3), 0)


@pytest.mark.parametrize("kind", SCALES)
def test_the_time_of_a_selection_does_not_depend_on_the_scale(kind):
    P, heads, k = 131040, 8, 96
    cfg = pkv.make_config(num_layers=1, num_q_heads=heads, num_kv_heads=heads, head_dim=64, window=ALPHA, pool_kernel=7, dtype="bf16",
                          avg_budget=ALPHA)
    ws = pkv.new_workspace(cfg, 1, P + ALPHA, DEV)
    idx = torch.empty(pkv.total_rows(cfg, k, [P + ALPHA]), dtype=torch.int32, device=DEV)

    def fastest(s):
        s, times = s[None].to(DEV), []
        for _ in range(20):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(10):
                pkv.select_topk(cfg, s, [P + ALPHA], k, idx, ws)
            b.record()
            b.synchronize()
            times.append(a.elapsed_time(b))
        return min(times)

    # a pass or two more over the candidates; with every position a candidate to the end it is 8 to 13 times as long
    assert fastest(scores_of(kind, heads, P, 3)) < 4 * fastest(scores_of("normal", heads, P, 3))


@pytest.mark.parametrize("P,budget", [(3000, 96), (9001, 2048), (40000, 1500)])
def test_the_fused_copy_places_every_listed_row(P, budget):
    """compress_layer (short lists: each CTA its own slice; long ones: dealt out evenly) and the paged call against the
    index list that they return."""
    heads, d, alpha, page = 2, 128, 8, 5
    lens = [P + alpha, P // 2]
    cfg = pkv.make_config(num_layers=1, num_q_heads=heads, num_kv_heads=heads, head_dim=d, window=alpha, pool_kernel=7, dtype="fp16",
                          avg_budget=budget)
    kl = pkv.layer_budgets(cfg)[0]
    g = torch.Generator(device=DEV).manual_seed(5)
    q = torch.randn(2, heads, alpha, d, generator=g, device=DEV).half()
    k, v = (torch.randn(2, heads, lens[0], d, generator=g, device=DEV).half() for _ in range(2))
    rows = pkv.total_rows(cfg, kl, lens)
    k_out, v_out = (torch.zeros(rows, d, dtype=torch.float16, device=DEV) for _ in range(2))
    idx, idx2 = (torch.zeros(rows, dtype=torch.int32, device=DEV) for _ in range(2))
    ws = pkv.new_workspace(cfg, 2, max(lens), DEV)
    pkv.compress_layer(cfg, 0, q, k, v, lens, k_out, v_out, idx, ws)
    pages = [pkv.pages_needed(cfg, kl, n, page) for n in lens]
    table = torch.randperm(heads * sum(pages), generator=torch.Generator().manual_seed(1)).to(torch.int32)
    k_pool, v_pool = (torch.zeros(heads * sum(pages), page, d, dtype=torch.float16, device=DEV) for _ in range(2))
    pkv.compress_layer_paged(cfg, 0, q, k, v, lens, table.to(DEV), k_pool, v_pool, idx2, ws)
    pkv.check_status(ws)
    assert torch.equal(idx, idx2)
    at, tab = 0, 0
    for b, n in enumerate(lens):
        c = pkv.kept_count(cfg, kl, n)
        for h in range(heads):
            pos = idx[at: at + c].long()
            assert torch.equal(pos[-alpha:].cpu(), torch.arange(n - alpha, n))
            slots = (table[tab: tab + pages[b]].long()[:, None] * page + torch.arange(page)).flatten()[:c].to(DEV)
            for src, packed, pool in ((k, k_out, k_pool), (v, v_out, v_pool)):
                assert torch.equal(packed[at: at + c], src[b, h][pos])
                assert torch.equal(pool.view(-1, d)[slots], src[b, h][pos])
            at += c
            tab += pages[b]

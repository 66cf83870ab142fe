"""The window-attention kernels at the edges of their split: CTAs dealt out to heads of one length (fewer tiles than CTAs, one
tile, whole and ragged last tiles), ranges that run over several heads and sequences, window rows around the two teams'
halves (16, 32, 48, 64 columns) and around 128, windows that do not divide a tile."""
import math

import pytest
import torch

import paper_2406_02069_b200 as pkv

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("group,heads,window,lens", [
    (4, 2, 32, [128]), (4, 3, 32, [129, 129]), (2, 8, 24, [1000]), (1, 5, 32, [3000]), (3, 2, 21, [700, 300]), (4, 80, 8, [300, 300]),
    (4, 40, 32, [700, 130, 512, 33]), (8, 2, 16, [2000]), (8, 3, 17, [513, 513]), (4, 9, 33, [640, 2111]), (5, 4, 48, [900]),
], ids=lambda v: str(v[0]) if isinstance(v, list) else str(v))
@pytest.mark.parametrize("dtype", ["bf16", "fp16"])
def test_scores_and_output(group, heads, window, lens, dtype):
    t = {"bf16": torch.bfloat16, "fp16": torch.float16}[dtype]
    cfg = pkv.make_config(num_layers=1, num_q_heads=group * heads, num_kv_heads=heads, head_dim=128, window=window, pool_kernel=1,
                          dtype=dtype, avg_budget=window)
    g = torch.Generator().manual_seed(51)
    q = (1.5 * torch.randn(len(lens), group * heads, window, 128, generator=g)).to(t)
    k, v = (torch.randn(len(lens), heads, max(lens), 128, generator=g).to(t) for _ in range(2))
    for b, n in enumerate(lens):
        k[b, :, n:], v[b, :, n:] = float("nan"), float("nan")
    ws = pkv.new_workspace(cfg, len(lens), max(lens), DEV)
    scores = torch.full((len(lens), heads, max(lens)), -1.0, device=DEV)
    out = torch.zeros(len(lens), group * heads, window, 128, device=DEV)
    pkv.attend_window(cfg, q.to(DEV), k.to(DEV), v.to(DEV), lens, out, scores, ws)
    pkv.check_status(ws)
    scores, out = scores.cpu().double(), out.cpu().double()
    eps = 4e-3 if dtype == "bf16" else 2.5e-3                # a weight's rounding to 16 bits and its exponential, 2e-3
    for b, n in enumerate(lens):
        P = n - window
        hidden = torch.arange(n)[None, :] > (P + torch.arange(window).repeat(group))[:, None]
        for h in range(heads):
            x = q[b, h * group:(h + 1) * group].double().reshape(-1, 128) @ k[b, h, :n].double().T / math.sqrt(128)
            w = torch.softmax(x.masked_fill(hidden, -math.inf), 1)
            want = w.sum(0)[:P] / group
            assert torch.all((scores[b, h, :P] - want).abs() <= 2e-3 * want + 1e-5), (b, h)
            assert torch.all(scores[b, h, P:] == -1.0)
            got = out[b, h * group:(h + 1) * group].reshape(-1, 128)
            assert torch.all((got - w @ v[b, h, :n].double()).abs() <= eps * (w @ v[b, h, :n].double().abs()) + 1e-6), (b, h)

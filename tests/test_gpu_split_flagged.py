"""fp32 scores where some or all tiles hold values that have no bfloat16 triples: such tiles are formed behind the others, into the
same logits and row statistics.  Row blocks, both head sizes, runs of a CTA over several heads and sequences, ragged ends."""
import math

import pytest
import torch

import paper_2406_02069_b200 as pkv

pytestmark = pytest.mark.gpu
DEV = "cuda"
REL = 2e-5                                                   # as in test_gpu_split.py


@pytest.mark.parametrize("group,heads,window,d,lens", [
    (4, 8, 32, 128, [4096 + 63]), (4, 2, 32, 128, [64, 65, 33, 127, 700]), (3, 3, 11, 64, [129, 1000]), (1, 2, 33, 128, [2049]),
    (8, 1, 40, 128, [777]), (5, 2, 52, 64, [513, 64]), (4, 40, 32, 64, [600, 65]),
], ids=lambda v: str(v[0]) if isinstance(v, list) else str(v))
@pytest.mark.parametrize("which", ["some keys", "all keys", "a window row", "all window rows"])
def test_scores_are_those_of_64_bit_arithmetic(group, heads, window, d, lens, which):
    """One channel of the keys times 2^100 and of the queries times 2^-100, or the other way round: the logits stay as they are."""
    g = torch.Generator().manual_seed(35)
    q = 1.5 * torch.randn(len(lens), group * heads, window, d, generator=g)
    k = torch.randn(len(lens), heads, max(lens), d, generator=g)
    if which.endswith("keys"):
        at = slice(7, None, 97) if which == "some keys" else slice(None)
        keep = torch.ones_like(k[..., 0], dtype=torch.bool)
        keep[:, :, at] = False
        k[..., 5] = torch.where(keep, torch.zeros(()), k[..., 5] * 2.0 ** 100)   # (the others have no share in the tiny channel)
        q[..., 5] *= 2.0 ** -100
    else:
        rows = slice(1, 2) if which == "a window row" else slice(None)
        q[:, :, rows, 5] *= 2.0 ** 100
        k[..., 5] *= 2.0 ** -100
        if which == "a window row":
            q[:, :, 0, 5] = q[:, :, 2:, 5] = 0.0
    exact_q, exact_k = q.double(), k.double()
    for b, n in enumerate(lens):
        k[b, :, n:] = float("nan")                           # rows behind a sequence are not read
    cfg = pkv.make_config(num_layers=1, num_q_heads=group * heads, num_kv_heads=heads, head_dim=d, window=window, pool_kernel=1,
                          dtype="fp32", avg_budget=window)
    ws = pkv.new_workspace(cfg, len(lens), max(lens), DEV)
    got = torch.full((len(lens), heads, max(lens)), -1.0, device=DEV)
    pkv.score_window(cfg, q.to(DEV), k.to(DEV), lens, got, ws)
    pkv.check_status(ws)
    got = got.cpu()
    for b, n in enumerate(lens):
        P = n - window
        hidden = torch.arange(n)[None, :] > (P + torch.arange(window).repeat(group))[:, None]
        for h in range(heads):
            x = exact_q[b, h * group:(h + 1) * group].reshape(-1, d) @ exact_k[b, h, :n].T / math.sqrt(d)
            want = torch.softmax(x.masked_fill(hidden, -math.inf), 1).sum(0)[:P] / group
            assert torch.all((got[b, h, :P].double() - want).abs() <= REL * want), (b, h)
            assert torch.all(got[b, h, P:] == -1.0)

"""Scores on the fp32 pipes at the edges of their tiles: window rows around the row blocks (32, 64, 128), one to many
key tiles, ragged batches, both head sizes, 16-bit inputs with more rows than the tensor-core path takes, and the three
ways through the kernels: logits kept in the workspace, formed again (the call without a workspace), and normalisers
handed in."""
import numpy as np
import pytest
import torch

import oracle
import paper_2406_02069_b200 as pkv
from helpers import assert_scores_close

pytestmark = pytest.mark.gpu
DEV = "cuda"

# (query heads per KV head, window, head size, dtype, lengths)
CASES = [
    (1, 3, 64, "fp32", [4, 5]), (2, 16, 128, "fp32", [128, 129, 17]), (1, 33, 128, "fp32", [300, 1000]), (4, 16, 64, "fp32", [64, 65, 511]),
    (5, 13, 128, "fp32", [777]), (4, 32, 128, "fp32", [2049, 640, 33]), (3, 43, 64, "fp32", [1500]), (8, 40, 128, "fp32", [600, 200]),
    (16, 17, 128, "bf16", [700, 90]), (9, 32, 64, "fp16", [513]),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "g%d_a%d_d%d_%s_n%d" % (c[0], c[1], c[2], c[3], c[4][0]))
def test_scores_against_the_oracle(case):
    group, window, d, dtype, lens = case
    heads = 2
    cfg = pkv.make_config(num_layers=1, num_q_heads=group * heads, num_kv_heads=heads, head_dim=d, window=window, pool_kernel=1,
                          dtype=dtype, avg_budget=window)
    t = {"fp32": torch.float32, "bf16": torch.bfloat16, "fp16": torch.float16}[dtype]
    g = torch.Generator().manual_seed(21)
    q = (1.5 * torch.randn(len(lens), group * heads, window, d, generator=g)).to(t)
    k = torch.randn(len(lens), heads, max(lens), d, generator=g).to(t)
    qd, kd = q.to(DEV), k.to(DEV)
    ws = pkv.new_workspace(cfg, len(lens), max(lens), DEV)
    kept, again, handed = (torch.full((len(lens), heads, max(lens)), -1.0, device=DEV) for _ in range(3))
    pkv.score_window(cfg, qd, kd, lens, kept, ws)
    pkv.score_window_static(cfg, qd, kd, lens, again)
    lse = torch.from_numpy(np.stack([oracle.window_lse(q[b], k[b, :, :n]) for b, n in enumerate(lens)]).astype(np.float32))
    pkv.score_window(cfg, qd, kd, lens, handed, ws, window_lse=lse.reshape(len(lens), group * heads, window).to(DEV))
    pkv.check_status(ws)
    for b, n in enumerate(lens):
        want, _ = oracle.window_scores(q[b], k[b, :, :n])
        want = want[0] if isinstance(want, tuple) else want
        P = n - window
        for got, what in ((kept, "kept"), (again, "again"), (handed, "handed")):
            # fp32 logits: |x| error below (d + 2) 2^-24 of the sum of |q k| terms (< 64 here), 5e-4 in the worst case; helpers'
            # 2e-3 relative bound covers it with the exponentials
            assert_scores_close(got[b, :, :P].cpu().numpy(), want, "%s sequence %d" % (what, b))
            assert torch.all(got[b, :, P:] == -1.0)          # nothing is written behind the prefix


def test_a_workspace_of_a_longer_context_serves_a_short_call():
    """Sized for a context whose logits are not kept, and cut down to what that call itself needs: with room for the short
    call's logits and without."""
    heads, group, window, d, n = 2, 4, 32, 128, 700
    cfg = pkv.make_config(num_layers=1, num_q_heads=group * heads, num_kv_heads=heads, head_dim=d, window=window, pool_kernel=1,
                          dtype="fp32", avg_budget=window)
    g = torch.Generator().manual_seed(22)
    q = 1.5 * torch.randn(1, group * heads, window, d, generator=g)
    k = torch.randn(1, heads, n, d, generator=g)
    want, _ = oracle.window_scores(q[0], k[0])
    ws = pkv.new_workspace(cfg, 1, 400000, DEV)
    assert ws.numel() > 256 << 20
    own = pkv.workspace_bytes(cfg, 1, n)
    for size in (ws.numel(), own, own - heads * group * window * 768 * 4):   # 768: n rounded up to whole tiles
        got = torch.full((1, heads, n), -1.0, device=DEV)
        pkv.score_window(cfg, q.to(DEV), k.to(DEV), [n], got, ws[:size])
        pkv.check_status(ws)
        assert_scores_close(got[0, :, : n - window].cpu().numpy(), want, "workspace of %d bytes" % size)
    with pytest.raises(pkv.PkvError):
        pkv.score_window(cfg, q.to(DEV), k.to(DEV), [n], got, ws[: own - heads * group * window * 768 * 4 - 256])

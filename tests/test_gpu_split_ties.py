"""fp32 scores: the same key in many tiles gets the same score bit for bit, whichever CTA has it and whatever its neighbours are
(far-away ones among them, whose exponentials are subnormal or zero), so that equal keys tie exactly."""
import pytest
import torch

import paper_2406_02069_b200 as pkv

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("group,window,d", [(4, 32, 128), (2, 20, 64), (5, 52, 128), (1, 32, 64)])
@pytest.mark.parametrize("ctas", [0, 7, 41])
def test_equal_keys_get_equal_scores(group, window, d, ctas):
    heads, lens = 5, [3000, 1500]
    cfg = pkv.make_config(num_layers=1, num_q_heads=group * heads, num_kv_heads=heads, head_dim=d, window=window, pool_kernel=1,
                          dtype="fp32", avg_budget=window, sweep_ctas=ctas)
    g = torch.Generator().manual_seed(37)
    q = 2.0 * torch.randn(len(lens), group * heads, window, d, generator=g)
    k = torch.randn(len(lens), heads, max(lens), d, generator=g)
    q[..., 0] = 16.0                                         # a channel that puts keys far below the others
    k[..., 0] = 0.0
    k[:, :, 5::128] = k[:, :, 5:6]
    for at, log2 in ((134, -100.0), (262, -135.0), (388, -160.0), (519, -128.0)):   # beside 133, 261, 389, 517
        k[:, :, at, 0] = log2 * d ** 0.5 * 0.6931 / 16.0
    ws = pkv.new_workspace(cfg, len(lens), max(lens), DEV)
    scores = torch.zeros(len(lens), heads, max(lens), device=DEV)
    pkv.score_window(cfg, q.to(DEV), k.to(DEV), lens, scores, ws)
    pkv.check_status(ws)
    for b, n in enumerate(lens):
        same = scores[b, :, 5: n - window: 128]
        assert torch.equal(same, same[:, :1].expand_as(same)), [int((row != row[0]).sum()) for row in same]

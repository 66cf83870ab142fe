"""pkv_config.sweep_ctas and the persistent sweep of fp32 scores: CTAs that go through many heads, row blocks and sequences."""
import math

import pytest
import torch

import paper_2406_02069_b200 as pkv

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _config(ctas, group, heads, window, d):
    return pkv.make_config(num_layers=1, num_q_heads=group * heads, num_kv_heads=heads, head_dim=d, window=window, pool_kernel=1,
                           dtype="fp32", avg_budget=window, sweep_ctas=ctas)


@pytest.mark.parametrize("ctas", [1, 7, 37, 74, 1024])
@pytest.mark.parametrize("group,heads,window,d,lens", [(4, 8, 32, 128, [2111, 700]), (5, 3, 40, 64, [1000, 65, 333])],
                         ids=["d128", "d64"])
def test_scores_are_those_of_64_bit_arithmetic(ctas, group, heads, window, d, lens):
    g = torch.Generator().manual_seed(36)
    q = 1.5 * torch.randn(len(lens), group * heads, window, d, generator=g)
    k = torch.randn(len(lens), heads, max(lens), d, generator=g)
    cfg = _config(ctas, group, heads, window, d)
    ws = pkv.new_workspace(cfg, len(lens), max(lens), DEV)
    got = torch.full((len(lens), heads, max(lens)), -1.0, device=DEV)
    pkv.score_window(cfg, q.to(DEV), k.to(DEV), lens, got, ws)
    pkv.check_status(ws)
    got = got.cpu()
    for b, n in enumerate(lens):
        P = n - window
        hidden = torch.arange(n)[None, :] > (P + torch.arange(window).repeat(group))[:, None]
        for h in range(heads):
            x = q[b, h * group:(h + 1) * group].double().reshape(-1, d) @ k[b, h, :n].double().T / math.sqrt(d)
            want = torch.softmax(x.masked_fill(hidden, -math.inf), 1).sum(0)[:P] / group
            assert torch.all((got[b, h, :P].double() - want).abs() <= 2e-5 * want), (b, h)   # as in test_gpu_split.py
            assert torch.all(got[b, h, P:] == -1.0)


def test_the_cap_holds():
    """8 heads of 16384 keys are 2048 tiles of more than a microsecond: one after the other in one CTA, a hundred times what the device
    takes with a CTA on every SM.  A sweep that ignores the cap takes the same time with and without."""
    group, heads, window, d, n = 4, 8, 32, 128, 16384
    q, k = torch.randn(1, group * heads, window, d, device=DEV), torch.randn(1, heads, n, d, device=DEV)
    scores = torch.zeros(1, heads, n, device=DEV)

    def milliseconds(ctas):
        cfg = _config(ctas, group, heads, window, d)
        ws = pkv.new_workspace(cfg, 1, n, DEV)
        best = math.inf
        for _ in range(5):
            start, end = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            start.record()
            pkv.score_window(cfg, q, k, [n], scores, ws)
            end.record()
            torch.cuda.synchronize()
            best = min(best, start.elapsed_time(end))
        pkv.check_status(ws)
        return best

    free, one, few = milliseconds(0), milliseconds(1), milliseconds(8)
    assert one > 8 * free and one > 3 * few > 3 * 2 * free, (free, few, one)

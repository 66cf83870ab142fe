"""The two-sweep score kernels at the edges of their split: window rows around the copies in the padding rows (32, 64), the
row blocks (128) and uneven halves, key tiles around 128 keys, and CTAs that go through many heads (one to three CTAs for all
of them), with the library's own normalisers and with the caller's."""
import numpy as np
import pytest
import torch

import oracle
import paper_2406_02069_b200 as pkv
from paper_2406_02069_b200 import binding
from helpers import assert_scores_close

pytestmark = pytest.mark.gpu
DEV = "cuda"

# (query heads per KV head, KV heads, window, head size, dtype, CTAs of a sweep or 0, lengths)
CASES = [
    (1, 3, 17, 128, "bf16", 1, [129, 128, 700]), (1, 2, 32, 64, "fp16", 2, [2000]), (3, 2, 11, 128, "bf16", 0, [500, 12]),
    (4, 2, 16, 64, "fp16", 3, [255, 256, 257, 18]), (5, 5, 13, 128, "bf16", 1, [400, 300]), (2, 8, 48, 128, "fp16", 3, [130, 1000, 600]),
    (4, 2, 32, 128, "bf16", 0, [3000]), (4, 3, 33, 128, "bf16", 1, [385, 90]), (8, 2, 23, 64, "fp16", 2, [640, 641]),
    (8, 4, 32, 128, "bf16", 3, [200, 1025, 129]),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "g%d_h%d_a%d_d%d_%s_c%d" % c[:6])
def test_scores_against_the_oracle(case):
    group, heads, window, d, dtype, ctas, lens = case
    cfg = pkv.make_config(num_layers=1, num_q_heads=group * heads, num_kv_heads=heads, head_dim=d, window=window, pool_kernel=1,
                          dtype=dtype, avg_budget=window, sweep_ctas=ctas)
    t = {"bf16": torch.bfloat16, "fp16": torch.float16}[dtype]
    g = torch.Generator().manual_seed(31)
    q = (2.0 * torch.randn(len(lens), group * heads, window, d, generator=g)).to(t)
    k = torch.randn(len(lens), heads, max(lens), d, generator=g).to(t)
    qd, kd = q.to(DEV), k.to(DEV)
    ws = pkv.new_workspace(cfg, len(lens), max(lens), DEV)
    own, handed = (torch.full((len(lens), heads, max(lens)), -1.0, device=DEV) for _ in range(2))
    lse = torch.from_numpy(np.stack([oracle.window_lse(q[b], k[b, :, :n]) for b, n in enumerate(lens)]).astype(np.float32))
    binding.test_hooks(two_sweeps=True)
    try:
        pkv.score_window(cfg, qd, kd, lens, own, ws)
        pkv.score_window(cfg, qd, kd, lens, handed, ws, window_lse=lse.reshape(len(lens), group * heads, window).to(DEV))
        pkv.check_status(ws)
    finally:
        binding.test_hooks()
    for b, n in enumerate(lens):
        want, _ = oracle.window_scores(q[b], k[b, :, :n])
        for got, what in ((own, "own"), (handed, "handed")):
            # exponentials to 7.5e-5 relative at most, fp32 sums: far inside the 2e-3 of the helper
            assert_scores_close(got[b, :, : n - window].cpu().numpy(), want, "%s sequence %d" % (what, b))
            assert torch.all(got[b, :, n - window:] == -1.0)


# (query heads per KV head, window, head size, dtype): 32, 64, 128 and 256 window rows
@pytest.mark.parametrize("ctas", [7, 20, 41, 0])
@pytest.mark.parametrize("group,window,d,dtype", [(4, 8, 128, "bf16"), (8, 8, 64, "fp16"), (4, 32, 128, "bf16"), (8, 32, 128, "fp16")])
def test_equal_keys_get_equal_scores_whichever_cta_has_them(group, window, d, dtype, ctas):
    """The same key in every tile of heads that many CTAs share, some of them as their second or third head: a head's row
    normalisers are the same bits in every CTA, so its equal keys tie exactly."""
    heads, lens = 5, [5000, 2100]
    cfg = pkv.make_config(num_layers=1, num_q_heads=group * heads, num_kv_heads=heads, head_dim=d, window=window, pool_kernel=1,
                          dtype=dtype, avg_budget=window, sweep_ctas=ctas)
    t = {"bf16": torch.bfloat16, "fp16": torch.float16}[dtype]
    g = torch.Generator().manual_seed(7)
    q = (2.0 * torch.randn(len(lens), group * heads, window, d, generator=g)).to(t)
    k = torch.randn(len(lens), heads, max(lens), d, generator=g).to(t)
    k[:, :, 5::128] = k[:, :, 5:6]
    ws = pkv.new_workspace(cfg, len(lens), max(lens), DEV)
    scores = torch.zeros(len(lens), heads, max(lens), device=DEV)
    binding.test_hooks(two_sweeps=True)
    try:
        pkv.score_window(cfg, q.to(DEV), k.to(DEV), lens, scores, ws)
        pkv.check_status(ws)
    finally:
        binding.test_hooks()
    for b, n in enumerate(lens):
        same = scores[b, :, 5: n - window: 128]
        assert torch.equal(same, same[:, :1].expand_as(same)), [int((row != row[0]).sum()) for row in same]


def test_a_long_sweep_ahead_is_not_a_wait_that_ran_out():
    """One CTA takes milliseconds for the row statistics of sixteen heads; the window-attention kernel behind it is on the
    device all that time, with the bound of its waits at about one millisecond (one head takes it less than half of that).
    Three attempts: a hiccup of the device may use up so short a bound, the sweep would do it every time."""
    heads, group, window, n = 16, 8, 32, 16384 + 32
    cfg = pkv.make_config(num_layers=1, num_q_heads=group * heads, num_kv_heads=heads, head_dim=128, window=window, pool_kernel=1,
                          dtype="bf16", avg_budget=window, sweep_ctas=1)
    g = torch.Generator(device=DEV).manual_seed(3)
    q = torch.randn(1, group * heads, window, 128, generator=g, device=DEV).bfloat16()
    k, v = (torch.randn(1, heads, n, 128, generator=g, device=DEV).bfloat16() for _ in range(2))

    def attend(bound):
        ws = pkv.new_workspace(cfg, 1, n, DEV)
        scores, out = torch.zeros(1, heads, n, device=DEV), torch.zeros(1, group * heads, window, 128, device=DEV)
        binding.test_hooks(wait_clocks=bound)
        try:
            pkv.attend_window(cfg, q, k, v, [n], out, scores, ws)
            pkv.check_status(ws)
        except pkv.PkvError:
            return None
        finally:
            binding.test_hooks()
        return scores, out

    want = attend(0)
    got = next((r for r in (attend(1 << 21) for _ in range(3)) if r is not None), None)
    assert got is not None, "the time of the sweep ahead counts as a wait"
    assert all(torch.equal(a, b) for a, b in zip(got, want))

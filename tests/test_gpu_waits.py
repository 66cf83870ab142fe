"""Waits that run out in the tensor-core kernels whose waits the other tests leave alone: the fp32 score kernel, and the
window-attention kernel for up to 128 window rows.  One K tile of one CTA is never handed over and the bound of the waits is
about a millisecond: the kernel winds down by itself, the status word says so, and the next call on the same workspace gives
what a fresh workspace gives."""
import pytest
import torch

import paper_2406_02069_b200 as pkv
from paper_2406_02069_b200 import binding

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("what,group,heads,window,n", [
    ("fp32", 4, 2, 32, 5000), ("fp32", 2, 3, 20, 300), ("fp32", 9, 2, 32, 1000),
    ("attend", 4, 2, 32, 5000), ("attend", 2, 3, 16, 1000), ("attend", 4, 2, 32, 160),
])
def test_a_wait_that_runs_out_is_reported(what, group, heads, window, n):
    dtype = {"fp32": torch.float32, "attend": torch.bfloat16}[what]
    cfg = pkv.make_config(num_layers=1, num_q_heads=group * heads, num_kv_heads=heads, head_dim=128, window=window, pool_kernel=1,
                          dtype={"fp32": "fp32", "attend": "bf16"}[what], avg_budget=window)
    g = torch.Generator(device=DEV).manual_seed(5)
    q = torch.randn(1, group * heads, window, 128, generator=g, device=DEV).to(dtype)
    k, v = (torch.randn(1, heads, n, 128, generator=g, device=DEV).to(dtype) for _ in range(2))

    def call(ws):
        scores, out = torch.zeros(1, heads, n, device=DEV), torch.zeros(1, group * heads, window, 128, device=DEV)
        if what == "fp32":
            pkv.score_window(cfg, q, k, [n], scores, ws)
        else:
            pkv.attend_window(cfg, q, k, v, [n], out, scores, ws)
        pkv.check_status(ws)
        return scores, out

    ws = pkv.new_workspace(cfg, 1, n, DEV)
    binding.test_hooks(wait_clocks=1 << 21, withhold_tile=what == "fp32", withhold_attend_tile=what == "attend")
    try:
        with pytest.raises(pkv.PkvError) as e:
            call(ws)
        assert e.value.status == binding.PKV_ERR_DEVICE_STATUS and "0x2" in str(e.value)
    finally:
        binding.test_hooks()
    ws[:256].zero_()
    again, fresh = call(ws), call(pkv.new_workspace(cfg, 1, n, DEV))
    assert all(torch.equal(a, b) for a, b in zip(again, fresh))

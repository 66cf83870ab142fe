"""Decode attention where warps and CTAs hold rows whose weights are 2^-130 of the largest: factors that are subnormal still count
where the values are large, and an infinity among them is an infinity."""
import math

import pytest
import torch

import paper_2406_02069_b200 as pkv

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("heads", [1, 40])                   # a cluster of CTAs to a head, and none
@pytest.mark.parametrize("dtype,value", [("fp32", 1e30), ("fp32", math.inf), ("bf16", math.inf), ("bf16", -math.inf)])
def test_rows_far_below_the_largest(dtype, value, heads):
    d, n, near = 128, 1024, 3
    t = {"fp32": torch.float32, "bf16": torch.bfloat16}[dtype]
    cfg = pkv.make_config(num_layers=1, num_q_heads=heads, num_kv_heads=heads, head_dim=d, window=1, pool_kernel=1, dtype=dtype,
                          avg_budget=1)
    q = torch.zeros(1, heads, d)
    q[..., 0] = 16.0
    k, v = torch.zeros(heads, n, d), torch.full((heads, n, d), 1e-10)
    k[:, :, 0] = -130.0 * math.sqrt(d) * math.log(2.0) / 16.0
    k[:, near, 0] = 0.0
    far = torch.arange(n) % 16 >= 8 if math.isfinite(value) else torch.arange(n) == n - 2
    v[:, far, 5] = value
    q, k, v = q.to(t), k.to(t), v.to(t)
    out = torch.zeros(1, heads, d, device=DEV)
    pkv.decode_attention(cfg, q.to(DEV), k.reshape(-1, d).to(DEV), v.reshape(-1, d).to(DEV), [n], n, out)
    w = torch.softmax((k.double() @ q[0].double().unsqueeze(-1)).squeeze(-1) / math.sqrt(d), 1)
    want = (w.unsqueeze(-1) * v.double()).sum(1)
    got = out[0].cpu().double()
    # a weight of 2^-130 is subnormal, 2^-149 apart: 1e-5 of it a step; the logits are 130 with 2^-22 of it off, 2e-5 of a weight
    at = want.isfinite()
    assert torch.equal(got[~at], want[~at])
    assert torch.all((got[at] - want[at]).abs() <= 1e-4 * want[at].abs())

"""fp32 scores from triples of bfloat16 on the tensor cores: edges of the key tiles (64) and row blocks (128), runs of a CTA
over several heads and sequences, scaled operands, and values that have no such triples."""
import math

import pytest
import torch

import paper_2406_02069_b200 as pkv

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _inputs(group, heads, window, d, lens, q_scale=1.0, k_scale=1.0):
    g = torch.Generator().manual_seed(31)
    q = 1.5 * q_scale * torch.randn(len(lens), group * heads, window, d, generator=g)
    k = k_scale * torch.randn(len(lens), heads, max(lens), d, generator=g)
    for b, n in enumerate(lens):
        k[b, :, n:] = float("nan")                           # rows behind a sequence are not read
    cfg = pkv.make_config(num_layers=1, num_q_heads=group * heads, num_kv_heads=heads, head_dim=d, window=window, pool_kernel=1,
                          dtype="fp32", avg_budget=window)
    return cfg, q, k


def _exact(cfg, q, k, lens):
    group, window = cfg.num_q_heads // cfg.num_kv_heads, cfg.window
    for b, n in enumerate(lens):
        P = n - window
        for h in range(cfg.num_kv_heads):
            x = q[b, h * group:(h + 1) * group].double().reshape(-1, cfg.head_dim) @ k[b, h, :n].double().T / math.sqrt(cfg.head_dim)
            hidden = torch.arange(n)[None, :] > (P + torch.arange(window).repeat(group))[:, None]
            yield b, h, P, torch.softmax(x.masked_fill(hidden, -math.inf), 1).sum(0)[:P] / group


def _run(cfg, q, k, lens):
    ws = pkv.new_workspace(cfg, len(lens), max(lens), DEV)
    got = torch.full((len(lens), cfg.num_kv_heads, max(lens)), -1.0, device=DEV)
    pkv.score_window(cfg, q.to(DEV), k.to(DEV), lens, got, ws)
    pkv.check_status(ws)
    return got.cpu()


# Logits (log2 units): sum |q k| is about 122 at d = 128, times log2(e) / sqrt(d) 16; a relative error of 2^-21 of that (24
# accumulations that cut off at 2^-23 of a partial sum, far smaller ones before them, and 2^-24 of the magnitudes for the
# products that are left out) is 7.4e-6.  It enters a score through
# its own logits and the normalisers: 2 x 7.4e-6 ln 2 and a few 2^-22 of the exponentials and sums, below 2e-5.
REL = 2e-5


@pytest.mark.parametrize("group,heads,window,d,lens", [
    (4, 8, 32, 128, [4096 + 63]), (4, 2, 32, 128, [64, 65, 33, 127, 128, 700]), (3, 3, 11, 64, [129, 1000]), (1, 2, 33, 128, [2049]),
    (4, 2, 40, 64, [640, 191]), (8, 1, 40, 128, [777]), (5, 2, 52, 128, [513, 64]), (4, 5, 32, 64, [3000, 65, 1500]),
], ids=lambda v: str(v[0]) if isinstance(v, list) else str(v))
def test_scores_are_those_of_64_bit_arithmetic(group, heads, window, d, lens):
    cfg, q, k = _inputs(group, heads, window, d, lens)
    got = _run(cfg, q, k, lens)
    for b, h, P, want in _exact(cfg, q, k, lens):
        assert torch.all((got[b, h, :P].double() - want).abs() <= REL * want), (b, h)
        assert torch.all(got[b, h, P:] == -1.0)              # nothing is written behind the prefix


# The large operand is beyond what is split (2^59); test_gpu_split_range.py has the powers around that
@pytest.mark.parametrize("power", [80, -80, 95, -95])
def test_operands_on_other_scales(power):
    lens = [300, 129]
    cfg, q, k = _inputs(4, 2, 32, 128, lens, 2.0 ** power, 2.0 ** -power)
    got = _run(cfg, q, k, lens)
    for b, h, P, want in _exact(cfg, q, k, lens):
        assert torch.all((got[b, h, :P].double() - want).abs() <= REL * want), (b, h)


@pytest.mark.parametrize("value", [math.inf, -math.inf, math.nan, 1e30])
def test_values_that_are_not_split(value):
    """A key of sequence 0, head 1 and a window row of sequence 1, head 0 with such a value: the logits, and with them the scores, are
    those of the multiply-adds that the call without a workspace uses; the other heads' scores are untouched."""
    lens = [400, 333]
    cfg, q, k = _inputs(4, 2, 32, 128, lens)
    k[0, 1, 70, 5] = value
    q[1, 2, 7, 9] = value
    got = _run(cfg, q, k, lens)
    ref = torch.full(got.shape, -1.0, device=DEV)
    pkv.score_window_static(cfg, q.to(DEV), k.to(DEV), lens, ref)
    ref = ref.cpu()
    assert torch.equal(got.isnan(), ref.isnan())
    at = ~ref.isnan()
    # (two fp32 evaluations of a logit: twice the bound above; scores far below the largest are sums of subnormal terms)
    assert torch.all((got[at] - ref[at]).abs() <= 2 * REL * ref[at].abs() + 1e-37)
    assert not got[0, 0, : 400 - 32].isnan().any() and not got[1, 1, : 333 - 32].isnan().any()

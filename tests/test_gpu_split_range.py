"""fp32 scores from triples of bfloat16 where products of finite operands leave the range of fp32: the logits, and with them the
scores, are those of the multiply-adds that the call without a workspace uses."""
import math

import pytest
import torch

import paper_2406_02069_b200 as pkv

pytestmark = pytest.mark.gpu
DEV = "cuda"
GROUP, HEADS, WINDOW, D, LENS, AT = 4, 2, 32, 128, [400, 333], 70
CFG = dict(num_layers=1, num_q_heads=GROUP * HEADS, num_kv_heads=HEADS, head_dim=D, window=WINDOW, pool_kernel=1, dtype="fp32",
           avg_budget=WINDOW)


def _inputs():
    g = torch.Generator().manual_seed(33)
    q = 1.5 * torch.randn(len(LENS), GROUP * HEADS, WINDOW, D, generator=g)
    k = torch.randn(len(LENS), HEADS, max(LENS), D, generator=g)
    return q, k


def _both(q, k):
    """Scores with stored logits and formed without them."""
    cfg = pkv.make_config(**CFG)
    ws = pkv.new_workspace(cfg, len(LENS), max(LENS), DEV)
    got, ref = (torch.zeros(len(LENS), HEADS, max(LENS), device=DEV) for _ in range(2))
    pkv.score_window(cfg, q.to(DEV), k.to(DEV), LENS, got, ws)
    pkv.score_window_static(cfg, q.to(DEV), k.to(DEV), LENS, ref)
    pkv.check_status(ws)
    return got.cpu(), ref.cpu()


def _same(got, ref):
    assert torch.equal(got.isnan(), ref.isnan())
    at = ~ref.isnan()
    # two evaluations of a logit, 2e-5 each (see test_gpu_split.py), and sums of subnormal terms
    assert torch.all((got[at] - ref[at]).abs() <= 4e-5 * ref[at].abs() + 1e-37)


# Magnitudes of the queries and of one key; the other keys are smaller by as much as the queries are larger
@pytest.mark.parametrize("q_power,key_power", [(70, 70), (50, 88), (40, 98), (58, 100), (100, 30), (64, 63), (62, 62)])
def test_a_logit_that_overflows_to_minus_infinity_takes_no_weight(q_power, key_power):
    q, k = _inputs()
    q = (q.abs() + 0.5) * 2.0 ** q_power
    k *= 2.0 ** -q_power
    k[0, 1, AT] = -(k[0, 1, AT].abs() * 2.0 ** q_power + 0.5) * 2.0 ** key_power
    got, ref = _both(q, k)
    assert got.isfinite().all() and got[0, 1, AT] == 0.0
    _same(got, ref)


# -2^70 (1 + 2^-7 - 2^-9): its high part is larger in magnitude, its middle part positive
@pytest.mark.parametrize("sign", [-1.0, 1.0])
def test_parts_of_opposite_signs(sign):
    q, k = _inputs()
    k[..., 5] = 0.0
    q[0, GROUP:, :, 5] = 2.0 ** 70
    k[0, 1, AT, 5] = sign * 2.0 ** 70 * (1 + 2.0 ** -7 - 2.0 ** -9)
    got, ref = _both(q, k)
    _same(got, ref)
    assert got[0, 0].isfinite().all() and got[1].isfinite().all()
    if sign < 0:
        assert got.isfinite().all() and got[0, 1, AT] == 0.0


@pytest.mark.parametrize("power", [58, 59, 60])
def test_around_the_magnitude_from_which_tiles_are_flagged(power):
    q, k = _inputs()
    q *= 2.0 ** power
    k *= 2.0 ** -power
    got, ref = _both(q, k)
    assert got.isfinite().all()
    _same(got, ref)
    assert math.isclose(got[0, 0].double().sum().item(), ref[0, 0].double().sum().item(), rel_tol=1e-5)

"""What the triples of bfloat16 behind the fp32 scores are worth: scores against 64 bits, closer than any kernel comes that leaves out
one of the six products.  The second half of that claim is checked on the CPU, with the products written out."""
import math

import pytest
import torch

CASES = [(4, 8, 32, 128, [4096 + 63]), (4, 2, 32, 128, [64, 65, 33, 127, 128, 700]), (3, 3, 12, 64, [129, 1000]), (1, 2, 33, 128, [2049]),
         (8, 1, 40, 128, [777]), (5, 2, 52, 128, [513, 64]), (4, 5, 32, 64, [3000, 65, 1500])]
# Largest relative error of a score.  An fp32 evaluation is off by some 2^-24 of a logit's sum of magnitudes and by a few 2^-24 of the
# normalisers, exponentials and sums; there is no useful bound on how these add up, so the figures are what one B200
# shows over the cases below, 8.2e-7, 5.4e-7 and 1.3e-6, doubled.  Without one of the products it is half as much again and more.
BOUND = {"dense": 1.6e-6, "one channel": 1.1e-6, "large last channel": 2.6e-6}


def _inputs(case, kind):
    group, heads, window, d, lens = case
    g = torch.Generator().manual_seed(38)
    q = 1.5 * torch.randn(len(lens), group * heads, window, d, generator=g)
    k = torch.randn(len(lens), heads, max(lens), d, generator=g)
    if kind == "one channel":
        q = torch.where(torch.arange(d) == 37, 6.0 * q, torch.zeros(()))
    elif kind == "large last channel":
        q[..., -1] *= 20.0
    return q, k


def _scores(logits, window, n):
    """Scores in 64 bits from the logits [rows][n] of a KV head."""
    rows, P = logits.shape[0], n - window
    hidden = torch.arange(n)[None, :] > (P + torch.arange(window).repeat(rows // window))[:, None]
    return torch.softmax(logits.masked_fill(hidden, -math.inf), 1).sum(0)[:P] * window / rows


def _heads(case, q, k):
    group, heads, window, d, lens = case
    for b, n in enumerate(lens):
        for h in range(heads):
            yield b, h, n, q[b, h * group:(h + 1) * group].reshape(-1, d), k[b, h, :n]


def _parts(x):
    high = x.bfloat16().float()
    mid = (x - high).bfloat16().float()
    return high, mid, (x - high - mid).bfloat16().float()


@pytest.mark.parametrize("kind", sorted(BOUND))
def test_six_products_are_inside_the_bound_and_fewer_are_not(kind):
    case = (4, 2, 32, 128, [700])
    q, k = _inputs(case, kind)
    for b, h, n, qh, kh in _heads(case, q, k):
        want = _scores(qh.double() @ kh.double().T / math.sqrt(128), 32, n)
        qp, kp = [p.double() for p in _parts(qh)], [p.double() for p in _parts(kh)]
        six = {(0, 0), (0, 1), (1, 0), (0, 2), (1, 1), (2, 0)}

        def error(products):
            x = sum(qp[i] @ kp[j].T for i, j in products) / math.sqrt(128)
            return ((_scores(x, 32, n) - want).abs() / want).max().item()
        assert error(six) < 0.2 * BOUND[kind]
        # (with one channel an error of a window row's value moves all its logits alike, which the normaliser takes out)
        for left_out in ({(0, 2), (2, 0)}, {(0, 2), (2, 0), (1, 1)}, {(0, 2)}, {(1, 1)}, {(0, 1)}) + (({(2, 0)},) if kind != "one channel" else ()):
            assert error(six - left_out) > 1.5 * BOUND[kind], left_out


@pytest.mark.gpu
@pytest.mark.parametrize("kind", sorted(BOUND))
@pytest.mark.parametrize("case", CASES, ids=lambda c: "g%d_h%d_a%d_d%d_n%d" % (*c[:4], c[4][0]))
def test_scores_are_those_of_64_bit_arithmetic(case, kind):
    import paper_2406_02069_b200 as pkv
    group, heads, window, d, lens = case
    q, k = _inputs(case, kind)
    cfg = pkv.make_config(num_layers=1, num_q_heads=group * heads, num_kv_heads=heads, head_dim=d, window=window, pool_kernel=1,
                          dtype="fp32", avg_budget=window)
    ws = pkv.new_workspace(cfg, len(lens), max(lens), "cuda")
    got = torch.zeros(len(lens), heads, max(lens), device="cuda")
    pkv.score_window(cfg, q.cuda(), k.cuda(), lens, got, ws)
    pkv.check_status(ws)
    got, worst = got.cpu().double(), 0.0
    for b, h, n, qh, kh in _heads(case, q, k):
        want = _scores(qh.double() @ kh.double().T / math.sqrt(d), window, n)
        worst = max(worst, ((got[b, h, : n - window] - want).abs() / want).max().item())
    print("largest relative error %.2e" % worst)
    assert worst <= BOUND[kind]

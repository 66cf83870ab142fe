"""The work a user of this framework has it do, as measurable cases through its public entry points.

Prefill side: compressing one layer (`compress_layer`), a whole model over a few streams
(`streaming.compress_model`), one layer into a paged pool with the normalisers handed over by the prefill attention
(`compress_layer_paged`), one layer together with the window rows' attention (`attend_compress_layer`), and the three
steps called one by one (`score_window`, `select_topk`, `gather_compact`).  Decode side: one new token through every
layer's compact cache, packed or paged (`decode_attention`, `decode_attention_paged`).

Inputs are those of `workloads.make_layer`: normal keys, queries that lean towards a few sink and needle keys, drawn
from the seed alone.  Everything else (sizes, lengths of the sequences, options) is in the case.
"""
import math
import random

import torch

import paper_2406_02069_b200 as pkv
from paper_2406_02069_b200 import streaming, workloads

WORD = {2: torch.int16, 4: torch.int32}


def _case(name, kind, heads, n, **more):
    """A case dict: heads = (query heads, KV heads, head size); n = (shortest, longest) sequence of the batch."""
    case = {"name": name, "kind": kind, "heads_q": heads[0], "heads_kv": heads[1], "dim": heads[2], "n_lo": n[0], "n_hi": n[1],
            "batch": 1, "lens_seed": 1, "dtype": "bf16", "window": 32, "pool": 7, "pool_kind": "max", "schedule": "linear",
            "budget": 128, "layers": 32, "layer": 8, "handoff": False, "page": 0, "streams": 1, "sweep_ctas": 0}
    case.update(more)
    return case


MHA, GQA4, GQA8 = (32, 32, 128), (32, 8, 128), (64, 8, 128)


def listed():
    return [
        # the smallest call: a toy model in fp32, as in a unit test or a notebook; latency is all there is
        _case("tiny_fp32_layer", "layer", (4, 2, 64), (512, 512), dtype="fp32", window=8, pool=5, budget=64, layers=2, layer=0),
        # an fp32 model (a numerics reference run) at a context that such runs use, of odd length
        _case("fp32_8k_layer", "layer", GQA4, (8101, 8101), dtype="fp32", budget=512),
        # a short chat context of a multi-head model: one layer, as an engine calls it at the end of that layer's prefill ...
        _case("llama2_7b_4k_layer", "layer", MHA, (4096, 4096)),
        # ... and all 32 layers after the prefill, spread over four streams
        _case("llama2_7b_4k_model", "model", MHA, (4096, 4096), streams=4),
        # a long document, grouped-query heads: one layer
        _case("llama3_8b_32k_layer", "layer", GQA4, (32768, 32768), budget=512),
        # the longest context: one layer
        _case("llama3_70b_128k_layer", "layer", GQA8, (131072, 131072), layers=80, layer=20),
        # a batch of eight requests of different lengths, all 32 layers: the most work a call is given
        _case("mistral_7b_ragged_model", "model", GQA4, (4096, 16384), batch=8, budget=512, streams=4, sweep_ctas=74),
        # a serving engine: paged cache, ragged batch, normalisers handed over by its prefill attention, fp16
        _case("mistral_7b_paged_handoff", "paged", GQA4, (4096, 16384), batch=8, budget=512, dtype="fp16", handoff=True, page=16),
        # the prefill leaves its last rows to this library: their attention output and the compressed layer from one call
        _case("llama3_8b_32k_attend", "attend", GQA4, (32768, 32768), budget=512),
        # the three steps one by one, head size 64, fp16, mean pool, two sequences of odd lengths
        _case("steps_fp16_d64_mean", "steps", (32, 8, 64), (7001, 10007), batch=2, dtype="fp16", pool=5, pool_kind="avg", budget=256, window=16),
        # decoding: one token of one sequence through all layers' packed caches with a large budget
        _case("decode_llama3_8b_b2048", "decode", GQA4, (32768, 32768), budget=2048),
        # decoding: one token of each of eight sequences through all layers' paged caches
        _case("decode_paged_mistral_7b", "decode", GQA4, (4096, 16384), batch=8, budget=512, page=16),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["layer", "layer", "layer", "fp32", "model", "paged", "attend", "steps", "decode", "decode"])
    if kind == "fp32":
        heads = rng.choice([(4, 2, 64), GQA4])
        n = _log_int(rng, 512, 8192)
        return _nameless(_case("", "layer", heads, (n, n), dtype="fp32", window=rng.choice([8, 16, 32]), pool=rng.choice([5, 7]),
                               budget=rng.choice([64, 128]), layers=rng.choice([2, 32]), layer=rng.choice([0, 1])))
    heads = rng.choice([MHA, GQA4, GQA4, GQA8] + ([(32, 8, 64)] if kind in ("layer", "steps", "decode") else []))
    layers = rng.choice([32, 80]) if kind in ("layer", "attend") else 32
    # tokens x KV heads (x layers of the pass) stay within the largest listed case of the kind
    room = {"layer": 131072 * 8, "attend": 32768 * 8, "steps": 2 * 16384 * 8, "paged": 8 * 16384 * 8, "model": 4 * 16384 * 8,
            "decode": 8 * 16384 * 8}[kind] // heads[1]
    batch = rng.choice([1, 1, 2, 3, 5, 8]) if kind != "steps" else rng.choice([1, 2])
    top = min(131072, room // batch)
    n_hi = _log_int(rng, 1024, top)
    n_lo = n_hi if batch == 1 else max(1024, n_hi // 4)
    budget = rng.choice([b for b in (64, 96, 128, 256, 512, 2048) if b * 4 <= n_lo])
    window = rng.choice([8, 16, 32]) if heads[0] // heads[1] == 8 else rng.choice([8, 16, 24, 32, 32, 48])
    window = min(window, budget // 2)
    case = _case("", kind, heads, (n_lo, n_hi), batch=batch, lens_seed=rng.randrange(1000), dtype=rng.choice(["bf16", "bf16", "fp16"]),
                 window=window, pool=rng.choice([5, 7]), pool_kind=rng.choice(["max", "max", "max", "avg"]),
                 schedule=rng.choice(["linear", "linear", "geometric"]), budget=budget, layers=layers, layer=rng.randrange(layers))
    if kind in ("layer", "model", "paged"):
        case["handoff"] = rng.random() < 0.25
    if kind == "paged" or (kind == "decode" and rng.random() < 0.5):
        case["page"] = rng.choice([16, 32, 64])
    if kind == "model":
        case["streams"] = rng.choice([1, 2, 4])
        case["sweep_ctas"] = 74 if case["streams"] == 4 and heads[0] != heads[1] else 0
    return _nameless(case)


def _nameless(case):
    del case["name"]
    return case


# ------------------------------------------------------------------------------------------------ sizes of a case
def _lens(case):
    r = random.Random(case["lens_seed"])
    return [r.randint(case["n_lo"], case["n_hi"]) for _ in range(case["batch"])]


def _cfg(case):
    return pkv.make_config(num_layers=case["layers"], num_q_heads=case["heads_q"], num_kv_heads=case["heads_kv"], head_dim=case["dim"],
                           window=case["window"], pool_kernel=case["pool"], dtype=case["dtype"], avg_budget=case["budget"],
                           pool_kind={"max": 0, "avg": 1}[case["pool_kind"]], schedule=case["schedule"],
                           inputs_final=case["kind"] == "model", sweep_ctas=case["sweep_ctas"])


def _workload(case, seed):
    return workloads.Workload("case", case["layers"], case["heads_q"], case["heads_kv"], case["dim"], case["batch"], case["n_lo"],
                              case["n_hi"], case["dtype"], case["window"], case["pool"], case["budget"], needles=8, seed=seed,
                              pool_kind=case["pool_kind"], schedule=case["schedule"])


def _pass_layers(case):
    """The layers one pass works on."""
    return list(range(case["layers"])) if case["kind"] in ("model", "decode") else [case["layer"]]


def work(case):
    cfg, lens = _cfg(case), _lens(case)
    budgets = pkv.layer_budgets(cfg)
    size = 4 if case["dtype"] == "fp32" else 2
    row = case["dim"] * size                                            # bytes of one key or value
    q_rows = case["heads_q"] * case["window"]                           # window rows of one sequence
    tokens = sum(lens)
    read = written = flops = 0
    for l in _pass_layers(case):
        kept = pkv.total_rows(cfg, budgets[l], lens)
        if case["kind"] == "decode":
            group = case["heads_q"] // case["heads_kv"]
            read += 2 * kept * row + len(lens) * case["heads_q"] * row
            written += len(lens) * case["heads_q"] * case["dim"] * 4
            flops += 4 * kept * group * case["dim"]
            continue
        read += tokens * case["heads_kv"] * row + len(lens) * q_rows * row + kept * row       # K, window queries, kept rows of V
        written += 2 * kept * row + 4 * kept                                                  # compact K and V, positions
        flops += 2 * tokens * q_rows * case["dim"]
        if case["handoff"]:
            read += 4 * len(lens) * q_rows
        if case["kind"] in ("attend", "steps"):
            written += 4 * (tokens - len(lens) * case["window"]) * case["heads_kv"]           # the scores
        if case["kind"] == "attend":
            read += tokens * case["heads_kv"] * row - kept * row                              # V whole
            written += 4 * len(lens) * q_rows * case["dim"]                                   # the attention output
            flops += 2 * tokens * q_rows * case["dim"]
    return {"bytes": read + written, "flops": flops}


def tolerance(case):
    if case["kind"] == "decode":
        return {"rel": 1e-5}                                            # fp32 sums over 16-bit rows
    # Copied rows and positions are whole values (rows are compared as bits); a position whose pooled score equals the
    # last kept one to rounding may differ, and then shifts the positions behind it.
    if case["kind"] == "attend":                                        # probabilities are rounded to the inputs' type
        return {"rel": 1e-2 if case["dtype"] == "bf16" else 2e-3, "differ": 0.01}
    if case["kind"] == "steps":
        return {"rel": 1e-4, "differ": 0.01}                            # scores: fp32 sums of approximated exponentials
    return {"differ": 0.01}


# ------------------------------------------------------------------------------------------------ inputs
def _window_lse(cfg, x, lens):
    """What a prefill attention holds for its last rows: the natural log of each row's softmax denominator."""
    group, window = cfg.num_q_heads // cfg.num_kv_heads, cfg.window
    out = torch.empty(x.q_win.shape[:3], dtype=torch.float32, device=x.q_win.device)
    for b, n in enumerate(lens):
        ahead = torch.arange(n, device=out.device)[None, :] - (n - window) > torch.arange(window, device=out.device)[:, None]
        for h in range(cfg.num_kv_heads):
            q = x.q_win[b, h * group:(h + 1) * group].float()
            logits = (q @ x.k[b, h, :n].float().T) / math.sqrt(cfg.head_dim)
            out[b, h * group:(h + 1) * group] = logits.masked_fill_(ahead, -math.inf).logsumexp(-1)
    return out


def _layer(case, cfg, seed, layer, lens):
    x = workloads.make_layer(_workload(case, seed), layer, device="cuda", seq_lens=lens)
    if case["handoff"]:
        x.window_lse = _window_lse(cfg, x, lens)
    return x


def _outputs(cfg, lens, rows, dtype):
    """Packed outputs of a list of layers in one allocation each, and a slice per layer."""
    total = sum(rows)
    k = torch.zeros(total, cfg.head_dim, dtype=dtype, device="cuda")
    v = torch.zeros_like(k)
    idx = torch.zeros(total, dtype=torch.int32, device="cuda")
    return (k, v, idx), [t.split(rows) for t in (k, v, idx)]


def _page_tables(cfg, budgets, lens, page, rng):
    """A pool's pages dealt out to the layers' block tables in random order, as an allocator in use would have them."""
    need = [cfg.num_kv_heads * sum(pkv.pages_needed(cfg, kl, n, page) for n in lens) for kl in budgets]
    order = torch.randperm(sum(need) + 7, generator=rng)[: sum(need)].to(torch.int32).cuda()
    return [t.contiguous() for t in order.split(need)], sum(need) + 7


def prepare(case, seed):
    cfg, lens = _cfg(case), _lens(case)
    layers = _pass_layers(case)
    budgets = [pkv.layer_budgets(cfg)[l] for l in layers]
    rows = [pkv.total_rows(cfg, kl, lens) for kl in budgets]
    dtype = {"fp32": torch.float32, "bf16": torch.bfloat16, "fp16": torch.float16}[case["dtype"]]
    rng = torch.Generator()
    rng.manual_seed(seed + 17)
    s = {"kind": case["kind"], "cfg": cfg, "lens": lens, "layers": layers, "budgets": budgets, "page": case["page"],
         "ws": pkv.new_workspace(cfg, len(lens), max(lens))}
    if case["kind"] == "decode":
        _prepare_decode(case, s, rows, dtype, rng)
        return s
    s["x"] = [_layer(case, cfg, seed, l, lens) for l in layers]
    whole, s["out"] = _outputs(cfg, lens, rows, dtype)
    s["result"] = [whole[0].view(WORD[dtype.itemsize]), whole[1].view(WORD[dtype.itemsize]), whole[2]]
    if case["kind"] in ("attend", "steps"):
        s["scores"] = torch.zeros(len(lens), cfg.num_kv_heads, max(lens) - cfg.window, device="cuda")
        s["result"].append(s["scores"])
    if case["kind"] == "attend":
        s["attn"] = torch.zeros(len(lens), cfg.num_q_heads, cfg.window, cfg.head_dim, device="cuda")
        s["result"].append(s["attn"])
    if case["kind"] == "model":
        m = streaming.LayerOutputs(cfg, lens, dtype)
        m.k, m.v, m.idx = s["out"]
        s["model"] = m
        s["streams"] = streaming.LayerStreams(cfg, lens, case["streams"]) if case["streams"] > 1 else None
    if case["kind"] == "paged":
        s["tables"], pages = _page_tables(cfg, budgets, lens, case["page"], rng)
        s["k_pool"] = torch.zeros(pages, case["page"], cfg.head_dim, dtype=dtype, device="cuda")
        s["v_pool"] = torch.zeros_like(s["k_pool"])
        s["result"] = [s["k_pool"].view(WORD[dtype.itemsize]), s["v_pool"].view(WORD[dtype.itemsize]), whole[2]]
    return s


def _prepare_decode(case, s, rows, dtype, rng):
    """Compact caches of every layer (kept keys: normal, the first ones of a head drawn towards the query) and a new
    token's queries per layer."""
    cfg, lens = s["cfg"], s["lens"]
    g = torch.Generator(device="cuda")
    g.manual_seed(rng.initial_seed())
    d = cfg.head_dim
    n_layers = len(s["layers"])
    s["pool"] = s["page"] > 0
    if s["pool"]:
        s["tables"], pages = _page_tables(cfg, s["budgets"], lens, s["page"], rng)
        s["caches"] = [torch.randn(pages, s["page"], d, generator=g, device="cuda").to(dtype) for _ in range(2)]
    else:
        s["caches"] = [t.split(rows) for t in (torch.randn(sum(rows), d, generator=g, device="cuda").to(dtype) for _ in range(2))]
    q = torch.randn(n_layers, len(lens), cfg.num_q_heads, d, generator=g, device="cuda")
    if not s["pool"]:
        toward = torch.nn.functional.normalize(torch.randn(d, generator=g, device="cuda"), dim=0)
        q += 4.0 * toward
        for l, kl in enumerate(s["budgets"]):
            at = 0
            for n in lens:
                count = pkv.kept_count(cfg, kl, n)
                heads = s["caches"][0][l][at: at + cfg.num_kv_heads * count].view(cfg.num_kv_heads, count, d)
                heads[:, :4] += (2.0 * math.sqrt(d) * toward).to(dtype)
                at += cfg.num_kv_heads * count
    s["q"] = [t for t in q.to(dtype)]
    whole = torch.zeros(n_layers, len(lens), cfg.num_q_heads, d, device="cuda")
    s["out"] = [t for t in whole]
    s["result"] = [whole]


# ------------------------------------------------------------------------------------------------ one pass
def run(s):
    kind, cfg, lens, ws = s["kind"], s["cfg"], s["lens"], s["ws"]
    if kind == "decode":
        for l, kl in enumerate(s["budgets"]):
            if s["pool"]:
                pkv.decode_attention_paged(cfg, s["q"][l], s["tables"][l], s["caches"][0], s["caches"][1], lens, kl, s["out"][l], ws)
            else:
                pkv.decode_attention(cfg, s["q"][l], s["caches"][0][l], s["caches"][1][l], lens, kl, s["out"][l])
        return s["result"]
    if kind == "model":
        streaming.compress_model(cfg, s["x"], lens, s["model"], ws, layer_streams=s["streams"])
        return s["result"]
    x, layer, kl = s["x"][0], s["layers"][0], s["budgets"][0]
    k_out, v_out, idx = (t[0] for t in s["out"])
    lse = getattr(x, "window_lse", None)
    if kind == "layer":
        pkv.compress_layer(cfg, layer, x.q_win, x.k, x.v, lens, k_out, v_out, idx, ws, window_lse=lse)
    elif kind == "paged":
        pkv.compress_layer_paged(cfg, layer, x.q_win, x.k, x.v, lens, s["tables"][0], s["k_pool"], s["v_pool"], idx, ws, window_lse=lse)
    elif kind == "attend":
        pkv.attend_compress_layer(cfg, layer, x.q_win, x.k, x.v, lens, s["attn"], k_out, v_out, idx, ws, scores=s["scores"])
    else:
        pkv.score_window(cfg, x.q_win, x.k, lens, s["scores"], ws)
        pkv.select_topk(cfg, s["scores"], lens, kl, idx, ws)
        pkv.gather_compact(cfg, x.k, x.v, idx, lens, kl, k_out, v_out)
    return s["result"]

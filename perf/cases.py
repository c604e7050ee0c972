"""The calls whose speed matters to a user of this library, over the range of sizes they come in.

A case is one call of a public entry point on seeded inputs: the decode-step attention over the
compressed cache (alone, together with the newest token's encode, with the BF16 window, for several
query tokens), the encoder (a prompt, the newest tokens) and the export of a cache to dequantised
values.  ``op`` names the call; the other fields are its shape and the options of its tables.

Values follow ``workloads``: keys N(0, 1) plus a per-(head, channel) offset, 1 % of the channels ten
times as large; values N(0, 1) or, with ``heavy_values``, Student-t with 5 degrees of freedom; queries
N(0, 1); everything rounded to bf16.  Pages of 16 tokens, in shuffled order.
"""
import random

import torch

import paper_2609_19880_b200 as dq
from paper_2609_19880_b200 import workloads

HEAD_DIM, PAGE, WINDOW = workloads.HEAD_DIM, workloads.PAGE, workloads.WINDOW
SM_SCALE = HEAD_DIM ** -0.5

# (query heads, KV heads) of the models in use: Llama-3-8B, Qwen2.5-7B, Llama-3-70B, Qwen2.5-14B,
# Qwen3-1.7B, Qwen2.5-1.5B, Qwen2.5-3B
MODELS = [(32, 8), (28, 4), (64, 8), (40, 8), (16, 8), (12, 2), (16, 2)]
ATTEND = ("attend", "step", "window", "speculate")
ENCODE = ("encode", "encode_new")

_DEFAULTS = dict(streams="head", bits=2.26, pairs=False, sigma=32, early_exit=False, heavy_values=False, rope=0, q_len=1,
                 resid=0, lens_seed=0)


def _case(name, op, batch, hq, hkv, ctx_min, ctx_max, **more):
    c = dict(_DEFAULTS, op=op, batch=batch, hq=hq, hkv=hkv, ctx_min=ctx_min, ctx_max=ctx_max)
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one chat session, short context: a call of a few microseconds of work, all latency and launches
        _case("attend_one_short", "attend", 1, 32, 8, 700, 700),
        # one layer of a decode step on a small server: two sequences, an odd GQA group of 7
        _case("step_two_sequences", "step", 2, 28, 4, 2571, 2571, heavy_values=True),
        # the layer of a decode step the library is quoted on: Llama-3-8B shape, batch 8, 8192 tokens
        _case("step_batch8_8k", "step", 8, 32, 8, 8192, 8192),
        # a loaded server: 128 sequences between 512 and 16384 tokens
        _case("attend_ragged_batch128", "attend", 128, 32, 8, 512, 16384, lens_seed=3),
        # one long document on a 70B model, at the largest bit budget (16 / 9 levels)
        _case("attend_long_4bit", "attend", 1, 64, 8, 131072, 131072, bits=4.0),
        # paired symbols, the variant that trades encode time for decode time, a medium ragged batch
        _case("attend_pairs_batch16", "attend", 16, 40, 8, 1900, 6100, pairs=True, lens_seed=5),
        # the paper's serving set-up: one stream per token over all heads, newest tokens in a BF16 window
        _case("window_token_streams", "window", 8, 32, 8, 8064, 8064, streams="token", resid=77),
        # speculative decoding: four query tokens per sequence against cache and window
        _case("speculate_four_tokens", "speculate", 4, 32, 8, 6016, 6016, q_len=4, resid=101),
        # a prompt batch: every key and value of 8 x 8192 tokens
        _case("encode_prompt", "encode", 8, 32, 8, 8192, 8192),
        # a prompt in the paper's grouping, keys handed over before their rotary embedding, ragged
        _case("encode_prompt_token_streams", "encode", 5, 32, 8, 1000, 4000, streams="token", rope=1, lens_seed=7),
        # the newest token of every sequence on its own (schedules that encode outside the decode step)
        _case("encode_newest_tokens", "encode_new", 24, 32, 8, 1000, 3000, lens_seed=9),
        # export of cached tokens to dequantised values (checks, migration to another cache)
        _case("export_cache", "export", 2, 32, 8, 3000, 5000, lens_seed=11),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    op = rng.choice(["attend", "attend", "step", "step", "window", "speculate", "encode", "encode", "encode_new", "export"])
    hq, hkv = rng.choice(MODELS)
    streams = "head" if op == "step" else rng.choice(["head", "head", "token"])
    more = dict(streams=streams, pairs=rng.random() < 0.25, early_exit=op in ENCODE and rng.random() < 0.2,
                heavy_values=rng.random() < 0.3, lens_seed=rng.randrange(1 << 20))
    if streams == "head":
        more["bits"] = rng.choice([2.26, 2.26, 2.26, 1.5, 2.0, 3.0] + ([] if more["pairs"] else [4.0]))
        more["sigma"] = 24 if rng.random() < 0.15 else 32
    if op == "encode":
        more["rope"] = rng.choice([0, 0, dq.ROPE_HALF, dq.ROPE_PAIRS])
    if op == "window":
        more["resid"] = rng.randint(1, WINDOW)
    if op == "speculate":
        more["q_len"] = rng.randint(2, 6)
        more["resid"] = rng.choice([0, rng.randint(8, WINDOW)])
    # the whole call, in (token, KV head) pairs, over its logarithm; the upper ends stay below the listed cases
    heavy = (2 if more["pairs"] else 1) * (2 if streams == "token" else 1) * (2 if more.get("bits", 0) >= 4.0 else 1)
    most = {"encode": 300_000 // heavy, "encode_new": 4_000, "export": 60_000}.get(op, 4_000_000 // more.get("q_len", 1))
    if op == "encode_new":
        batch = max(1, _log_uniform(rng, 8, most) // hkv)
        ctx = rng.randint(200, 4000)
        return _case(None, op, min(batch, 500), hq, hkv, ctx, ctx + rng.randint(0, ctx), **more)
    tokens = max(64, _log_uniform(rng, 512 * hkv, most) // hkv)
    batch = min(_log_uniform(rng, 1, 128), max(1, tokens // 100))
    ctx = min(131072, max(33, tokens // batch))
    spread = rng.choice([0.0, rng.random() * 0.9])
    return _case(None, op, batch, hq, hkv, max(1, int(ctx * (1 - spread))), max(1, int(ctx * (1 + spread))), **more)


def _lens(case):
    r = random.Random(case["lens_seed"])
    return [r.randint(case["ctx_min"], case["ctx_max"]) for _ in range(case["batch"])]


def _records(case):
    """(record bytes, levels) of keys and values."""
    if case["streams"] == "token":   # 335 / 235 bytes for 1024 values, 8 / 6 levels
        hs = case["hkv"]
        return (335 * hs // 8, 8), (235 * hs // 8, 6)
    k_rec, v_rec, k_lev, v_lev = workloads.BUDGETS[case["bits"]]
    return (k_rec, k_lev), (v_rec, v_lev)


def _stream_heads(case):
    return case["hkv"] if case["streams"] == "token" else 1


def _tables(case):
    hs, out = _stream_heads(case), []
    for i, (rec, levels) in enumerate(_records(case)):
        out.append(dq.dq_build_tables(levels, rec * 8 / (HEAD_DIM * hs), alpha=1.4, has_mean=i == 0, rotate=True,
                                      heads_per_stream=hs, drift_early_exit=case["early_exit"],
                                      sigma_bits=case["sigma"], pair_symbols=case["pairs"]))
    return out


def _containers(case, num_pages, rec):
    hkv, hs = case["hkv"], _stream_heads(case)
    shape = (num_pages, hkv, PAGE, rec) if hs == 1 else (num_pages, 1, (rec + 3) // 4, PAGE, 4)
    return torch.zeros(shape, dtype=torch.uint8, device="cuda")


def prepare(case, seed):
    lens = _lens(case)
    (k_rec, k_lev), (v_rec, v_lev) = _records(case)
    cfg = workloads.Config("case", case["batch"], case["hq"], case["hkv"], lens, seed, k_rec, v_rec, k_lev, v_lev,
                           shuffle_pages=True, v_student_t=case["heavy_values"])
    w = workloads.generate(cfg, device="cuda")
    tk, tv = _tables(case)
    hkv, batch, hq, q_len = case["hkv"], case["batch"], case["hq"], case["q_len"]
    s = {"op": case["op"], "hkv": hkv, "tk": tk, "tv": tv, "k_cont": _containers(case, w.num_pages, k_rec),
         "v_cont": _containers(case, w.num_pages, v_rec), "page_table": w.page_table, "seq_lens": w.seq_lens,
         "mean_q": torch.zeros((batch, w.max_windows, hkv, HEAD_DIM), dtype=torch.int8, device="cuda"),
         "mean_scale": torch.zeros((batch, w.max_windows, hkv), dtype=torch.float32, device="cuda"), "rope": None}
    if case["op"] == "encode":
        s.update(k=w.k, v=w.v, seq_id=w.seq_id, pos=w.pos, slot=w.slot)
        if case["rope"]:
            freq = 10000.0 ** (-torch.arange(HEAD_DIM // 2, device="cuda", dtype=torch.float64) / (HEAD_DIM // 2))
            ang = torch.arange(max(lens), device="cuda", dtype=torch.float64)[:, None] * freq
            s["rope"] = (ang.cos().float(), ang.sin().float(), case["rope"])
        return s
    # every other call works on a cache that holds its tokens
    dq.dq_encode_tokens(tk, tv, w.k, w.v, w.seq_id, w.pos, w.slot, s["k_cont"], s["v_cont"], s["mean_q"], s["mean_scale"])
    last = torch.cumsum(torch.tensor(lens), 0).cuda() - 1
    if case["op"] in ("step", "encode_new"):
        s.update(k=w.k[last].contiguous(), v=w.v[last].contiguous(), seq_id=w.seq_id[last].contiguous(),
                 pos=w.pos[last].contiguous(), slot=w.slot[last].contiguous())
    if case["op"] == "export":
        s.update(seq_id=w.seq_id, pos=w.pos, slot=w.slot)
        for kind in "kv":
            s["symbols_" + kind] = torch.zeros((len(w.pos), hkv, HEAD_DIM), dtype=torch.uint8, device="cuda")
            s["dequant_" + kind] = torch.zeros((len(w.pos), hkv, HEAD_DIM), dtype=torch.float32, device="cuda")
    if case["op"] in ATTEND:
        gen = torch.Generator(device="cuda").manual_seed(seed + 1)
        rows = (batch, q_len, hq, HEAD_DIM) if case["op"] == "speculate" else (batch, hq, HEAD_DIM)
        s["q"] = torch.randn(rows, generator=gen, device="cuda").bfloat16()
        s["out"] = torch.zeros_like(s["q"])
        per_pass = min(q_len, 8 // (hq // hkv))
        nbytes = dq.dq_decode_workspace_bytes(batch, hq * per_pass, w.page_table.shape[1])
        s["workspace"] = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        s["resid"] = (None, None, None)
        if case["resid"]:
            rk, rv = workloads.make_kv(cfg, batch * WINDOW, gen, "cuda", w.k_offsets, w.k_gain)
            shape = (batch, WINDOW, hkv, HEAD_DIM)
            fill = torch.full((batch,), case["resid"], dtype=torch.int32, device="cuda")
            s["resid"] = (rk.view(shape), rv.view(shape), fill)
    return s


def run(s):
    op = s["op"]
    cache = (s["k_cont"], s["v_cont"], s["mean_q"], s["mean_scale"])
    if op == "attend":
        dq.dq_decode_attention(s["tk"], s["tv"], s["q"], *cache, s["page_table"], s["seq_lens"], s["hkv"], SM_SCALE, s["out"],
                               s["workspace"])
    elif op == "step":
        dq.dq_decode_step(s["tk"], s["tv"], s["k"], s["v"], s["slot"], s["q"], *cache, s["page_table"], s["seq_lens"], s["hkv"],
                          SM_SCALE, s["out"], s["workspace"])
        return {"out": s["out"], "k_cont": s["k_cont"], "v_cont": s["v_cont"], "mean_q": s["mean_q"]}
    elif op == "window":
        dq.dq_decode_attention_residual(s["tk"], s["tv"], s["q"], *cache, s["page_table"], s["seq_lens"], *s["resid"], s["hkv"],
                                        SM_SCALE, s["out"], s["workspace"])
    elif op == "speculate":
        rk, rv, rl = s["resid"]
        dq.dq_decode_attention_multi(s["tk"], s["tv"], s["q"], *cache, s["page_table"], s["seq_lens"], s["hkv"], SM_SCALE,
                                     s["out"], s["workspace"], resid_k=rk, resid_v=rv, resid_lens=rl)
    elif op in ENCODE:
        mode = dq.MEAN_COMPUTE if op == "encode" else dq.MEAN_REUSE
        dq.dq_encode_tokens(s["tk"], s["tv"], s["k"], s["v"], s["seq_id"], s["pos"], s["slot"], *cache, mode, rope=s["rope"])
        return dict(zip(("k_cont", "v_cont", "mean_q", "mean_scale"), cache))
    else:
        dq.dq_decode_tokens(s["tk"], s["k_cont"], s["slot"], s["hkv"], s["symbols_k"], s["dequant_k"], s["mean_q"],
                            s["mean_scale"], s["seq_id"], s["pos"])
        dq.dq_decode_tokens(s["tv"], s["v_cont"], s["slot"], s["hkv"], s["symbols_v"], s["dequant_v"])
        return {k: s[k] for k in ("symbols_k", "dequant_k", "symbols_v", "dequant_v")}
    return s["out"]


def work(case):
    """Bytes every implementation reads or writes once, and the arithmetic of the contractions (attention),
    of the rotation and of the least-squares sums (encoder), or of the affine map (export)."""
    lens = _lens(case)
    hq, hkv, batch, hs = case["hq"], case["hkv"], case["batch"], _stream_heads(case)
    (k_rec, _), (v_rec, _) = _records(case)
    windows = sum((n + WINDOW - 1) // WINDOW for n in lens) * hkv * (HEAD_DIM + 4)
    tokens = batch if case["op"] == "encode_new" else sum(lens)
    values = tokens * hkv * HEAD_DIM
    records = tokens * (hkv // hs) * (k_rec + v_rec)
    if case["op"] in ENCODE:
        rope = 2 * 4 * (HEAD_DIM // 2) * max(lens) if case["rope"] else 0
        means = batch * hkv * (HEAD_DIM + 4) if case["op"] == "encode_new" else windows
        return {"bytes": 2 * 2 * values + records + means + rope + 12 * tokens, "flops": 2 * values * (7 + 4)}
    if case["op"] == "export":
        return {"bytes": records + windows + 12 * tokens + 2 * (1 + 4) * values, "flops": 2 * 3 * values}
    q_len, resid = case["q_len"], case["resid"]
    io = 2 * 2 * batch * q_len * hq * HEAD_DIM + 2 * 2 * batch * resid * hkv * HEAD_DIM
    if case["op"] == "step":
        io += 2 * 2 * batch * hkv * HEAD_DIM
    pages = 4 * sum((n + PAGE - 1) // PAGE for n in lens)
    return {"bytes": records + windows + pages + io, "flops": 4 * HEAD_DIM * hq * q_len * (tokens + batch * resid)}


def tolerance(case):
    # attention: binary32 sums over fp16 hi + lo operands, stored as bf16 (an element on a rounding edge moves by
    # one bf16 step, 2^-8); records, means, symbols and dequantised values are defined bit for bit
    return {"rel": 2e-3, "max": 0.1} if case["op"] in ATTEND else "exact"

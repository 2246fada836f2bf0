"""What a user of the pipelined decoder has it do, as cases that can be timed and compared.

A decode takes the encoder memory of a batch of sequences and gives the token streams of their
subsequences; around it stand the one-pass scoring of given targets, a serving loop that admits the
next sequence of a queue into a row that has become free, and the stand-alone operators.  Shapes are those
of the five seeded workloads (phrase-level targets = many short subsequences, sentence-level
targets = few long ones, over a long context), plus one request alone, and everything between.

Weights are drawn at the workloads' scale, with two differences that make the streams reproducible: the
context projections are wide enough for cross-attention to single out positions, as it does in a trained model, and
the vocabulary projection prefers one successor of every token by a clear margin, so that rounding does
not decide which token follows.  Lengths are given (the workloads' distributions), and a decode ends at a step
budget (time_max) near the end of its longest subsequences: its last step still has rows, whose logits or
final hidden states come back beside the tokens.
"""
import math

import numpy as np
import torch

from paper_2506_23431_b200 import binding as B
from paper_2506_23431_b200 import workload as W

# vocabulary sizes and widths of the workloads
_BART = {"layers": 6, "heads": 12, "vocab": 50265}
_T5 = {"layers": 12, "heads": 16, "vocab": 32128}


def _decode(name, model, batch, ctx, sub_max, delta_t, lengths, steps, pos, **kw):
    c = {"name": name, "kind": "decode", **model, "batch": batch, "ctx": ctx, "ragged": False, "sub_max": sub_max, "delta_t": delta_t,
         "lengths": lengths, "steps": steps, "pos": pos, "dtype": "bf16", "kv8": False, "logits": False, "host": False}
    c.update(kw)
    return c


def listed():
    return [
        # a unit-test sized model in fp32, one sequence: launches and latency are all there is
        _decode("tiny_fp32", {"layers": 2, "heads": 4, "vocab": 8192}, 1, 256, 4, 2, "uniform:8:16", 20, "t5", dtype="fp32", logits=True),
        # one document of odd length for one interactive user
        _decode("one_request", _BART, 1, 777, 8, 3, "lognormal:3.0:0.4:48", 40, "rope", logits=True),
        # a batch of documents, sentences of every length, logits wanted beside the tokens
        _decode("bart_base", _BART, 16, 1024, 8, 3, "geometric:20:48", 48, "rope", logits=True),
        # keyphrases of many documents, from host memory to host memory
        _decode("keyphrase_host", _BART, 64, 1024, 32, 1, "uniform:3:8", 36, "rope", host=True),
        # few long documents
        _decode("long_context", _T5, 8, 4096, 8, 4, "uniform:16:40", 60, "t5"),
        # summarisation of a batch of documents: the largest decode
        _decode("summarisation", _T5, 32, 2048, 16, 2, "lognormal:3.0:0.4:64", 56, "t5"),
        # the same with the projected context stored in 8 bits, documents of different lengths
        _decode("summarisation_kv8", _T5, 32, 2048, 16, 2, "lognormal:3.0:0.4:64", 56, "t5", kv8=True, ragged=True),
        # a server: a queue of documents through the rows of a running batch
        _decode("serving", _BART, 16, 1024, 8, 3, "geometric:20:48", 120, "rope", kind="serve", queue=40, ragged=True),
        # scoring of given summaries in one pass (re-ranking, perplexity)
        _decode("score", _T5, 32, 2048, 16, 2, "lognormal:3.0:0.4:64", 256, "t5", kind="score"),
        # scoring with the logits of every position (distillation), few documents
        _decode("score_logits", _BART, 3, 1000, 8, 3, "geometric:20:48", 128, "rope", kind="score", logits=True, ragged=True),
        # the operators alone, inside somebody else's model
        {"name": "op_cross_attention", "kind": "cross", "heads": 12, "batch": 16, "ctx": 1000, "rows": 9, "dtype": "bf16"},
        {"name": "op_vocab_argmax", "kind": "vocab", "heads": 12, "rows": 100, "vocab": 50265},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["decode", "decode", "decode", "decode", "decode", "serve", "score", "cross", "vocab"])
    heads = rng.choice([4, 8, 12, 16])
    if kind == "cross":
        return {"kind": "cross", "heads": heads, "batch": _log_int(rng, 1, 64), "ctx": _log_int(rng, 64, 4096), "rows": rng.randint(1, 32),
                "dtype": rng.choice(["bf16", "bf16", "bf16", "fp32"])}
    if kind == "vocab":
        return {"kind": "vocab", "heads": heads, "rows": _log_int(rng, 1, 600), "vocab": _log_int(rng, 1000, 50265)}
    dtype = rng.choice(["bf16"] * 5 + ["fp32"]) if kind == "decode" else "bf16"
    layers = rng.randint(2, 12)
    ctx = _log_int(rng, 64, 4096)
    most = {"decode": 64, "serve": 24, "score": 32}[kind] if dtype == "bf16" else 4
    sub_max, delta_t = _log_int(rng, 1, 32), rng.randint(1, 4)
    cap = rng.choice([8, 16, 40, 48, 64])
    # no more context, and no more target rows in one scoring pass, than the largest listed case
    batch = min(_log_int(rng, 1, most), max(1, (16 if kind == "serve" else 32) * 12 * 2048 * 16 // (layers * ctx * heads)))
    if kind == "score":
        batch = min(batch, max(1, 16000 // (sub_max * cap)))
    lengths = rng.choice(["uniform:%d:%d" % (max(1, cap // 3), cap), "geometric:%d:%d" % (max(2, cap // 2), cap), "lognormal:%.2f:0.4:%d" % (math.log(cap / 2.6), cap)])
    steps = max(8, min(64, (sub_max - 1) * delta_t + (cap * 3) // 4))
    kv8 = dtype == "bf16" and rng.random() < 0.25
    if kv8:
        ctx = max(64, ctx // 16 * 16)
    c = _decode("", {"layers": layers, "heads": heads, "vocab": _log_int(rng, 1000, 50265)}, batch, ctx, sub_max, delta_t, lengths, steps,
                rng.choice(["t5", "rope"]), kind=kind, dtype=dtype, kv8=kv8, ragged=rng.random() < 0.5)
    # 8-bit context and the one-pass scoring take at most 32 open subsequences per sequence; so does everything drawn here
    if kind == "decode":
        c["logits"] = batch * min(sub_max, cap // delta_t + 1) * c["vocab"] < 30_000_000 and rng.random() < 0.4
        c["host"] = rng.random() < 0.3
    if kind == "score":
        c["steps"] = 256
        c["logits"] = batch * sub_max * cap * c["vocab"] < 200_000_000 and rng.random() < 0.5
    if kind == "serve":
        c["steps"], c["queue"] = 96, 2 * batch
    del c["name"]
    return c


# ---- shapes -------------------------------------------------------------------------------------------------
def _workload(c, seed):
    parts = c["lengths"].split(":")
    dist = (parts[0],) + tuple(float(p) if "." in p else int(p) for p in parts[1:])
    cap = int(dist[-1])
    # a row that is taken again starts its own clock, so a server's step budget is that of one sequence
    t_max = 128 if c["kind"] == "serve" else c["steps"]
    return W.Workload("case", c["layers"], 64 * c["heads"], c["heads"], 256 * c["heads"], c["vocab"], c["dtype"], c["batch"], c["ctx"],
                      c["sub_max"], c["delta_t"], t_max, cap, dist, W.POS_T5_BIAS if c["pos"] == "t5" else W.POS_ROPE, seed,
                      kv_c_dtype="e4m3" if c["kv8"] else "same")


def _queue(c):
    return c.get("queue", c["batch"])


# ---- inputs -------------------------------------------------------------------------------------------------
def _weights(w, gen):
    d, ff, v = w.d_model, w.d_ff, w.vocab

    def normal(std, *shape):
        return torch.randn(*shape, generator=gen, device="cuda") * std

    out = {"embed": normal(1.0, v, d)}
    for l in range(w.n_layers):
        for name, rows, cols, std in (("wqkv", d, 3 * d, 0.03), ("wo", d, d, 0.02), ("wq_c", d, d, 0.05), ("wkv_c", d, 2 * d, 0.05),
                                      ("wo_c", d, d, 0.02), ("w1", d, ff, 0.02), ("w2", ff, d, 0.02)):
            out[f"l{l}.{name}"] = normal(std * math.sqrt(1024 / rows) if name != "w2" else std * math.sqrt(4096 / rows), rows, cols)
        for name in ("norm1", "norm2", "norm3"):
            out[f"l{l}.{name}"] = 1 + normal(0.1, d)
    out["final_norm"] = 1 + normal(0.1, d)
    # successor of token order[i] = order[i + 1]; the three special ids follow nothing
    order = torch.randperm(v - 3, generator=gen, device="cuda") + 3
    lm_head = normal(0.02, v, d)
    lm_head[order[1:]] = 0.02 * out["embed"][order[:-1]]
    lm_head[order[0]] = 0.02 * out["embed"][w.bos_id]
    out["lm_head"] = lm_head
    out["rel_bias"] = normal(w.rel_bias_std, w.n_heads, w.rel_buckets)
    return {k: t.cpu().numpy() for k, t in out.items()}


def _documents(c, w, gen):
    """Encoder memory of every sequence [n, ctx, d], context lengths, subsequence lengths."""
    n = _queue(c)
    # targets that are scored have the lengths of the case, whatever their words (the outputs keep their shape)
    lengths_of = w.scaled(batch=n, seed=0) if c["kind"] == "score" else w.scaled(batch=n)
    mem = torch.randn(n, w.ctx, w.d_model, generator=gen, device="cuda").to(torch.bfloat16 if w.dtype == "bf16" else torch.float32)
    return mem, W.make_ctx_len(lengths_of, ragged=c["ragged"]), W.make_forced_len(lengths_of)


def prepare(case, seed):
    c = dict(case)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    if c["kind"] == "cross":
        dt = torch.bfloat16 if c["dtype"] == "bf16" else torch.float32
        b, h, ctx, rows = c["batch"], c["heads"], c["ctx"], c["rows"]
        q = (1.5 * torch.randn(b, rows, 64 * h, generator=gen, device="cuda")).to(dt)
        kv = torch.randn(b, h, 2, ctx, 64, generator=gen, device="cuda").to(dt)
        n_rows = torch.full((b,), rows, dtype=torch.int32, device="cuda")
        ctx_len = torch.randint(ctx // 2, ctx + 1, (b,), generator=gen, device="cuda", dtype=torch.int32)
        return {"kind": "cross", "q": q, "kv": kv, "n_rows": n_rows, "ctx_len": ctx_len}
    if c["kind"] == "vocab":
        d = 64 * c["heads"]
        return {"kind": "vocab", "hidden": torch.randn(c["rows"], d, generator=gen, device="cuda").bfloat16(),
                "lm_head": (0.02 * torch.randn(c["vocab"], d, generator=gen, device="cuda")).bfloat16()}
    w = _workload(c, seed)
    mem, ctx_len, forced = _documents(c, w, gen)
    dec = B.PipelinedDecoder(w.hyper(), _weights(w, gen), c["batch"], store_logits=c["logits"] and c["kind"] == "decode")
    s = {"kind": c["kind"], "case": c, "w": w, "dec": dec, "ctx_len": ctx_len, "forced": forced}
    if c["kind"] == "score":
        # targets of the drawn lengths, random content
        toks = W.make_random_tokens(w, (c["batch"], c["sub_max"], w.max_sub_len))
        s["targets"] = [[toks[b, i, :forced[b, i]].tolist() for i in range(c["sub_max"])] for b in range(c["batch"])]
    if c["host"]:
        s["mem"] = mem.cpu().pin_memory()
    elif c["kind"] == "serve":
        s["mem"], s["first"] = [m.contiguous() for m in mem], mem[: c["batch"]].contiguous()
    else:
        s["mem"] = mem
    return s


# ---- one pass -----------------------------------------------------------------------------------------------
def _hidden(s):
    """The residual stream behind the last layer after the last step, [rows, d_model]."""
    dec, d = s["dec"], s["w"].d_model
    rows = dec.batch * dec.rows_per_seq
    return dec.debug_read(B.PD_BUF_X, np.float32, rows * d).reshape(rows, d)


def _run_decode(s):
    dec = s["dec"]
    if s["case"]["host"]:
        out = dec.generate_host(s["mem"], s["ctx_len"], s["forced"])
    else:
        dec.encode_context(s["mem"], s["ctx_len"], s["forced"])
        dec.run()
        out = dec.collect()
    if s["case"]["logits"]:
        out["logits"], out["row_sub"] = dec.get_logits()
    else:
        out["hidden"] = _hidden(s)
    return out


def _run_serve(s):
    dec, c, w = s["dec"], s["case"], s["w"]
    batch, queue = c["batch"], c["queue"]
    tokens = np.full((queue, w.sub_max, w.max_sub_len), -1, np.int32)
    lens = np.zeros((queue, w.sub_max), np.int32)
    steps = np.zeros((queue,), np.int32)
    holds, nxt = list(range(batch)), batch
    dec.encode_context(s["first"], s["ctx_len"][:batch], s["forced"][:batch])
    for t in range(c["steps"]):
        dec.step()
        if t % 4 != 3:
            continue
        done, _ = dec.rows_done()
        for row in range(batch):
            if not done[row] or holds[row] < 0:
                continue
            got, doc = dec.collect_row(row), holds[row]
            tokens[doc], lens[doc], steps[doc] = got["tokens"], got["lens"], got["steps"]
            holds[row] = -1
            if nxt < queue:
                dec.admit(row, s["mem"][nxt], int(s["ctx_len"][nxt]), s["forced"][nxt])
                holds[row], nxt = nxt, nxt + 1
        if all(h < 0 for h in holds):
            break
    return {"tokens": tokens, "lens": lens, "steps": steps, "open": dec.collect(), "hidden": _hidden(s)}


def _run_score(s):
    dec = s["dec"]
    dec.encode_context(s["mem"], s["ctx_len"], s["forced"])
    logprob, loss, logits = dec.teacher_forward(s["targets"], want_logits=s["case"]["logits"])
    out = {"logprob": logprob, "loss": loss}
    if logits is not None:
        out["logits"] = logits
    return out


def run(state):
    if state["kind"] == "cross":
        return B.cross_attention(state["q"], state["kv"], state["n_rows"], state["ctx_len"], 0.125, splits=2)
    if state["kind"] == "vocab":
        return B.vocab_argmax(state["hidden"], state["lm_head"], want_logits=True)
    return {"decode": _run_decode, "serve": _run_serve, "score": _run_score}[state["kind"]](state)


# ---- what a pass cannot do without --------------------------------------------------------------------------
def _schedule(c, w, forced, n_steps):
    """Per step of one sequence on its own clock: (open subsequences, cache entries visible to the last of them)."""
    per = []
    for t in range(1, n_steps + 1):
        rows = entries = 0
        upto = 0
        for i in range(w.sub_max):
            age = t - (i * w.delta_t + 1)                 # content tokens it has at step t
            if age < 0:
                break
            upto += min(age, int(forced[i])) + 1
            if age <= forced[i]:
                rows, entries = rows + 1, upto
        if rows == 0:                                     # every subsequence held has ended: the sequence stops
            break
        per.append((rows, entries))
    return per


def work(case):
    c = dict(case)
    if c["kind"] == "cross":
        e, d = (2 if c["dtype"] == "bf16" else 4), 64 * c["heads"]
        keys = 0.75 * c["batch"] * c["ctx"]
        return {"bytes": keys * 2 * d * e + 2 * c["batch"] * c["rows"] * d * e, "flops": 4 * keys * c["rows"] * d}
    if c["kind"] == "vocab":
        d = 64 * c["heads"]
        return {"bytes": c["vocab"] * d * 2 + c["rows"] * (d * 2 + c["vocab"] * 4 + 8), "flops": 2 * c["rows"] * d * c["vocab"]}
    w = _workload(c, 0)
    n = _queue(c)
    many = w.scaled(batch=n)
    ctx_len, forced = W.make_ctx_len(many, ragged=c["ragged"]).astype(np.int64), W.make_forced_len(many)
    e, d, L = (2 if c["dtype"] == "bf16" else 4), w.d_model, w.n_layers
    kv_e = 1 if c["kv8"] else e
    per_layer = 6 * d * d + 2 * d * w.d_ff                 # q k v, o, cross q, cross o, feed-forward
    keys = int(ctx_len.sum())
    # the context: encoder memory in, keys and values of every layer out
    byt = keys * d * e + L * 2 * d * d * e + keys * L * 2 * d * kv_e
    flops = 4 * keys * d * d * L
    if c["kind"] == "score":
        rows = int((forced + 1).sum())
        per_seq = (forced + 1).sum(axis=1)
        byt += (L * per_layer + 2 * w.vocab * d) * e + keys * L * 2 * d * kv_e + rows * 4 + (rows * w.vocab * 4 if c["logits"] else 0)
        flops += 2 * rows * (L * per_layer + w.vocab * d) + 4 * d * L * int((per_seq * ctx_len).sum()) + 2 * d * L * int((per_seq * per_seq).sum())
        return {"bytes": float(byt), "flops": float(flops)}
    n_steps = w.time_max
    runs = [_schedule(c, w, forced[b], n_steps) for b in range(n)]
    longest = max(len(r) for r in runs) if c["kind"] == "decode" else c["steps"]
    rows = sum(r for run_ in runs for r, _ in run_)
    byt += longest * (L * per_layer + w.vocab * d) * e     # every weight once per step
    flops += 2 * rows * (L * per_layer + w.vocab * d)
    for b, run_ in enumerate(runs):
        live = sum(1 for r, _ in run_ if r > 0)
        seen = sum(v for r, v in run_ if r > 0)
        byt += L * 2 * d * (live * int(ctx_len[b]) * kv_e + seen * e)
        flops += 4 * d * L * sum(r * (int(ctx_len[b]) + v) for r, v in run_)
    last = sum(r[-1][0] for r in runs if r)
    byt += last * (w.vocab if c["logits"] else d) * 4
    return {"bytes": float(byt), "flops": float(flops)}


def tolerance(case):
    if case["kind"] == "vocab":
        return {"rel": 1e-5, "max": 1e-4, "differ": 0.01}
    if case["kind"] == "cross":
        return {"rel": 1e-2 if case["dtype"] == "bf16" else 1e-5}
    if case["dtype"] == "fp32":
        return {"rel": 1e-5}
    # bf16 decodes against fp32 decodes with the same (bf16-representable) weights and inputs: rel 0.0042 to 0.0047,
    # largest difference 0.038 to 0.072 of the root mean square; token streams, lengths, flags and steps the same
    return {"rel": 2e-2, "max": 0.3}

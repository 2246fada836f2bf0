"""Small decodes, forwards and operator calls at the edges of the kernels' tiles and of the rules that choose between
kernels, against the CPU oracle on the same seeded inputs.  Tolerances: the decode and forward bars of the other GPU tests
(1e-4 fp32, 2e-2 bf16 on logits of this scale); the operator's follow from its roundings, stated beside them."""
import numpy as np
import pytest

from paper_2506_23431_b200 import workload as W
from tests import parity
from tests.test_gpu_kernels import cross_case, oracle_cross
from tests.test_gpu_parity import check
from tests.test_gpu_teacher_forward import run_case

pytestmark = pytest.mark.gpu

BASE = dict(d_model=192, n_heads=3, n_layers=2, vocab=515, norm_gain_std=0.1, ctx=150, delta_t=1)
T5, ROPE = W.POS_T5_BIAS, W.POS_ROPE

DECODES = [
    # storage, sequences, open rows per sequence, inner width, positions, longest subsequence, 8-bit context
    ("bf16", 1, 1, 264, ROPE, 30, False),      # one row; an inner width that ends inside a 32-wide K unit
    ("bf16", 1, 16, 1024, T5, 20, False),      # one full 16-row tile; the longest reduction that one CTA takes
    ("bf16", 1, 17, 1048, ROPE, 20, False),    # one row in the second tile; a reduction over two CTAs, the second nearly empty
    ("bf16", 3, 11, 520, T5, 14, True),        # sequences that share a row tile; 8-bit context
    ("bf16", 4, 32, 2056, ROPE, 34, False),    # 128 rows: the most that run packed; three CTAs per reduction
    ("bf16", 4, 32, 264, T5, 34, True),        # the same with two query tiles per sequence over 8-bit context
    ("bf16", 3, 43, 264, T5, 45, False),       # 129 rows and more than 32 in a sequence: the kernels beyond
    ("bf16", 5, 26, 264, ROPE, 28, False),     # 130 rows, unpacked, two query tiles
    ("fp32", 1, 1, 264, ROPE, 30, False),
    ("fp32", 1, 16, 1024, T5, 20, False),
    ("fp32", 1, 17, 1032, ROPE, 20, False),    # second row tile, second chunk of attention rows, reduction over two CTAs
    ("fp32", 2, 16, 520, T5, 18, False),       # 32 rows: the most that the fp32 products take
    ("fp32", 3, 11, 264, ROPE, 14, False),     # 33 rows: library products
    ("fp32", 1, 64, 264, T5, 66, False),       # four chunks of attention rows
]


@pytest.mark.parametrize("dtype,batch,rows,d_ff,pos,length,kv8", DECODES)
def test_decode_at_row_and_reduction_edges(dtype, batch, rows, d_ff, pos, length, kv8):
    base = W.CONFIGS["tiny" if dtype == "fp32" else "bart_base"]
    # subsequences long enough for `rows` of them to be open at once; a few steps beyond that are compared
    wl = base.scaled(name="edges", batch=batch, sub_max=rows, d_ff=d_ff, pos_mode=pos, max_sub_len=length, time_max=min(rows + 6, 96),
                     length_dist=("uniform", max(1, length - 4), length), kv_c_dtype="e4m3" if kv8 else "same",
                     **dict(BASE, ctx=144 if kv8 else 150))
    s = check(wl, rows=[0, batch - 1] if batch > 1 else None, ragged=True, free_run=False)
    assert s["max_err"] < parity.TOL[dtype]


CROSS = [
    # sequences, rows, heads, ctx -> CTAs per (sequence, head)
    (1, 16, 18, 1300),     # 8, eleven tiles over eight CTAs
    (1, 17, 18, 900),      # 8, two query tiles: fifteen records in the first CTA's ring
    (1, 3, 19, 1300),      # 4
    (37, 5, 1, 300),       # 4 by the segments, 2 by the three tiles
    (38, 32, 1, 700),      # 2, two query tiles
    (75, 1, 1, 520),       # 1, one tile beyond a multiple of the ring
    (300, 2, 2, 40),       # more sequences than a launch once took
    (2, 9, 2, 128),        # one tile exactly
    (2, 9, 2, 129),        # and one key more
]


@pytest.mark.parametrize("batch,rows,heads,ctx", CROSS)
def test_cross_attention_at_cluster_edges(batch, rows, heads, ctx):
    """Unused rows come back as zeros and the status word clear, whatever the scratch held; two launches agree bit for bit."""
    import torch
    from paper_2506_23431_b200 import binding as B
    q, kv, n_rows, ctx_len = cross_case(31, batch, rows, heads, ctx, "bf16")
    ref = oracle_cross(q, kv, n_rows, ctx_len, heads, 0.125)
    dev = torch.device("cuda", 0)
    args = (torch.from_numpy(q).to(dev, torch.bfloat16), torch.from_numpy(kv).to(dev, torch.bfloat16),
            torch.from_numpy(n_rows).to(dev), torch.from_numpy(ctx_len).to(dev), 0.125, 1)
    scratch = torch.full((B.cross_attention_scratch_bytes(batch, rows, heads, 1),), 0x5a, dtype=torch.uint8, device=dev)
    out = B.cross_attention(*args, scratch)
    again = B.cross_attention(*args, scratch)
    torch.cuda.synchronize()
    assert int(scratch[:16].view(torch.int32)[2]) == 0
    assert torch.equal(out.view(torch.int16), again.view(torch.int16))
    got = out.float().cpu().numpy().astype(np.float64)
    # weights and result are rounded to bf16 (2^-9 each, relative) and a row of weights sums to 1: twice 2^-9 of the largest value
    assert np.abs(got - ref).max() <= 2 * 2.0 ** -9 * max(1.0, np.abs(kv[np.isfinite(kv)]).max())


@pytest.mark.parametrize("rows,d_model,vocab", [(128, 64, 227), (129, 128, 451), (256, 64, 230)])
def test_vocab_logits_at_row_tile_edges(rows, d_model, vocab):
    """Both row-tile variants of the kernel, vocabularies whose logit rows start off every 16-byte boundary."""
    import torch
    from paper_2506_23431_b200 import binding as B
    g = np.random.Generator(np.random.Philox(key=np.array([rows, vocab], dtype=np.uint64)))
    hidden = W.bf16_round(g.standard_normal((rows, d_model), dtype=np.float32))
    lm_head = W.bf16_round(0.05 * g.standard_normal((vocab, d_model), dtype=np.float32))
    ref = hidden.astype(np.float64) @ lm_head.astype(np.float64).T
    dev = torch.device("cuda", 0)
    ids, best, logits = B.vocab_argmax(torch.from_numpy(hidden).to(dev, torch.bfloat16), torch.from_numpy(lm_head).to(dev, torch.bfloat16), want_logits=True)
    got = logits.cpu().numpy()
    # fp32 accumulation of d_model exact products: d_model * 2^-23 of the sum of their magnitudes
    tol = d_model * 2.0 ** -23 * (np.abs(hidden).astype(np.float64) @ np.abs(lm_head).astype(np.float64).T).max()
    assert np.abs(got - ref).max() <= tol
    assert (ids.cpu().numpy() == got.argmax(axis=1)).all() and (best.cpu().numpy() == got.max(axis=1)).all()


FORWARDS = [
    # sequences, subsequences, longest, heads, vocabulary, positions, context
    (3, 4, 15, 2, 301, ROPE, 131),     # up to 64 rows a sequence: one block of 64; logit rows off the 16-byte boundary; three keys in a second tile
    (2, 5, 25, 2, 302, T5, 128),       # several blocks of 64, the last one partly filled; one context tile exactly
    (2, 5, 25, 2, 302, T5, 65),        # one key in the second half of a tile
    (2, 2, 25, 2, 302, ROPE, 1),       # a context of one key
    (12, 16, 40, 6, 303, T5, 131),     # enough blocks of 128 rows to fill the GPU
    (12, 16, 40, 6, 304, ROPE, 400),   # more tiles than the ring holds
]


@pytest.mark.parametrize("batch,sub_max,length,heads,vocab,pos,ctx", FORWARDS)
def test_teacher_forward_at_block_edges(batch, sub_max, length, heads, vocab, pos, ctx):
    wl = W.CONFIGS["bart_base"].scaled(name="tf_edges", n_layers=1, d_model=64 * heads, n_heads=heads, d_ff=256, vocab=vocab, norm_gain_std=0.1,
                                       batch=batch, ctx=ctx, sub_max=sub_max, delta_t=2, max_sub_len=length,
                                       length_dist=("uniform", max(0, length - 6), length), time_max=sub_max * 2 + length, pos_mode=pos)
    assert run_case(wl, 2e-2) < 2e-2


def test_teacher_forward_when_the_running_maximum_moves():
    """Sharp cross-attention: scores with a spread of several powers of two, so that rows meet larger ones tile after tile and what they
    have summed is rescaled.  Queries and keys rounded to bf16 (2^-9 each) leave scores of up to 15 off by 0.06 at most, weights and
    the layer's output off by as much relatively; the output projection takes that below the usual bar."""
    from oracle import pipelined_decoder as O
    from paper_2506_23431_b200.binding import PipelinedDecoder
    from tests.test_gpu_teacher_forward import targets_of
    wl = W.CONFIGS["bart_base"].scaled(name="tf_sharp", n_layers=1, d_model=128, n_heads=2, d_ff=256, vocab=300, norm_gain_std=0.1, batch=2, ctx=700,
                                       sub_max=5, delta_t=2, max_sub_len=25, length_dist=("uniform", 15, 25), time_max=35, pos_mode=ROPE)
    weights, mem, ctx_len = W.make_weights(wl), W.make_encoder_memory(wl), W.make_ctx_len(wl, ragged=True)
    for name in ("l0.wq_c", "l0.wkv_c"):
        weights[name] = W.bf16_round(7 * weights[name])
    subs = targets_of(wl)
    dec = PipelinedDecoder(wl.hyper(), weights, wl.batch)
    dec.encode_context(dec.device_memory(mem), ctx_len, None)
    logits = dec.teacher_forward(subs, want_logits=True)[2].cpu().numpy().astype(np.float64)
    orc = O.PipelinedDecoderOracle(weights, wl.hyper())
    ref = np.concatenate([orc.teacher_forward(mem[b], int(ctx_len[b]), subs[b])["logits"] for b in range(wl.batch)])
    assert np.abs(logits - ref).max() <= 2e-2
    dec.close()


@pytest.mark.parametrize("ctx", [65, 700])
def test_teacher_forward_when_one_warp_of_a_block_lags(ctx):
    """Rows of one 32-row group meet a larger score half after half (their keys grow along the context) and rescale what they have summed;
    the other groups' queries are near zero and never do: the groups of a block drift apart.  Repeats agree bit for bit, and the oracle's
    forward within the bar of the test above (two halves: the shortest context with a hand-over)."""
    from oracle import pipelined_decoder as O
    from paper_2506_23431_b200.binding import PipelinedDecoder
    wl = W.CONFIGS["bart_base"].scaled(name="tf_lag", n_layers=1, d_model=128, n_heads=2, d_ff=256, vocab=300, norm_gain_std=0.0, batch=8, ctx=ctx,
                                       sub_max=5, delta_t=2, max_sub_len=31, length_dist=("uniform", 31, 31), time_max=42, pos_mode=ROPE)
    weights, mem, ctx_len = W.make_weights(wl), W.make_encoder_memory(wl), np.full(wl.batch, ctx, np.int32)
    # words 3 .. 149 live in the first half of the columns, the others and <bos> in the second; only the first half makes queries
    g = np.random.Generator(np.random.Philox(key=np.array([ctx, 77], dtype=np.uint64)))
    embed = g.standard_normal((300, 128), dtype=np.float32)
    embed[3:150, 64:] = 0
    embed[:3, :64] = 0
    embed[150:, :64] = 0
    weights["embed"] = W.bf16_round(embed)
    weights["l0.wq_c"][64:] = 0
    for name in ("l0.wq_c", "l0.wkv_c"):
        weights[name] = W.bf16_round(8 * weights[name])
    mem = W.bf16_round(mem * np.linspace(0.1, 1.3, ctx, dtype=np.float32)[None, :, None])
    words = g.integers(150, 300, size=(wl.batch, 5, 31))
    for b in range(wl.batch):
        words[b, b % 4] = g.integers(3, 150, size=31)          # rows 32 i .. 32 i + 31 are subsequence i + 1's (31 words and <bos>)
    subs = words.tolist()
    dec = PipelinedDecoder(wl.hyper(), weights, wl.batch)
    dec.encode_context(dec.device_memory(mem), ctx_len, None)
    runs = [dec.teacher_forward(subs, want_logits=True)[2].cpu().numpy() for _ in range(12)]
    orc = O.PipelinedDecoderOracle(weights, wl.hyper())
    for r in runs[1:]:
        assert np.array_equal(r, runs[0])
    rows = 5 * 32
    for b in (0, 1, 2, 3):
        ref = orc.teacher_forward(mem[b], ctx, subs[b])["logits"]
        assert np.abs(runs[0][b * rows:(b + 1) * rows] - ref).max() <= 2e-2
    dec.close()


@pytest.mark.parametrize("vocab", [301, 304])
def test_teacher_forward_into_a_slice_of_a_larger_buffer(vocab):
    """The caller's logits start at any float: rows of a larger buffer, one to three floats off a 16-byte boundary.  The same rows through
    another order of fp32 sums: 300 terms, 300 x 2^-24 relative of a log-probability of a few units; the logits 128 terms of products."""
    import ctypes as C

    import torch
    from paper_2506_23431_b200 import binding as B
    from tests.test_gpu_teacher_forward import targets_of
    wl = W.CONFIGS["bart_base"].scaled(name="tf_slice", n_layers=1, d_model=128, n_heads=2, d_ff=256, vocab=vocab, norm_gain_std=0.1, batch=2, ctx=96,
                                       sub_max=4, delta_t=2, max_sub_len=15, length_dist=("uniform", 5, 15), time_max=25, pos_mode=ROPE)
    subs = targets_of(wl)
    dec = B.PipelinedDecoder(wl.hyper(), W.make_weights(wl), wl.batch)
    dec.encode_context(dec.device_memory(W.make_encoder_memory(wl)), W.make_ctx_len(wl), None)
    lp, loss, want = dec.teacher_forward(subs, want_logits=True)
    rows = len(lp)
    n_sub = np.array([len(s) for s in subs], np.int32)
    lens, toks = np.zeros((wl.batch, wl.sub_max), np.int32), np.zeros((wl.batch, wl.sub_max, wl.max_sub_len), np.int32)
    for b, seq in enumerate(subs):
        for i, sub in enumerate(seq):
            lens[b, i], toks[b, i, :len(sub)] = len(sub), sub
    nbytes = int(B._lib.pd_teacher_forward_scratch_bytes(dec._h, rows, 0))
    scratch = torch.empty(nbytes, dtype=torch.uint8, device=dec.device)
    for off in (1, 2, 3):
        buf = torch.full((off + (rows + 1) * vocab,), 7.0, device=dec.device)
        torch.cuda.synchronize()
        got_lp, n, got_loss = np.empty(rows, np.float32), C.c_int32(0), C.c_double(0.0)
        st = B._lib.pd_teacher_forward(dec._h, B._p(n_sub), B._p(lens), B._p(toks), None, C.c_void_p(scratch.data_ptr()), C.c_size_t(nbytes),
                                       got_lp.ctypes.data_as(C.POINTER(C.c_float)), C.c_void_p(buf.data_ptr() + 4 * off), C.byref(n), C.byref(got_loss))
        assert st == 0 and n.value == rows
        got = buf[off:off + rows * vocab].reshape(rows, vocab)
        assert (got - want).abs().max().item() <= 1e-4
        assert (buf[:off] == 7).all() and (buf[off + rows * vocab:] == 7).all()          # nothing beside the slice
        assert np.abs(got_lp - lp).max() <= 1e-4 and abs(got_loss.value - loss) <= 1e-4 * rows
    dec.close()


@pytest.mark.parametrize("dtype,batch", [("bf16", 2), ("bf16", 20), ("fp32", 2), ("fp32", 5)])
def test_embedding_and_gains_that_start_at_any_value(dtype, batch):
    """embed and every norm gain one value into larger buffers, on the packed, the library and both fp32 paths of a step and in the one-pass
    forward: the same bits as from tables of their own."""
    import ctypes as C

    import torch
    from paper_2506_23431_b200 import binding as B
    wl = W.CONFIGS["tiny" if dtype == "fp32" else "bart_base"].scaled(
        name="tables", batch=batch, n_layers=2, d_model=128, n_heads=2, d_ff=256, vocab=301, norm_gain_std=0.1, ctx=96, sub_max=7, delta_t=2,
        max_sub_len=15, length_dist=("uniform", 5, 15), time_max=26, pos_mode=ROPE)
    mem, ctx_len, forced = W.make_encoder_memory(wl), W.make_ctx_len(wl), W.make_forced_len(wl)
    subs = [[[5, 6, 7 + b], [8, 9]] for b in range(batch)]
    dec = B.PipelinedDecoder(wl.hyper(), W.make_weights(wl), wl.batch, store_logits=True)

    def results():
        dec.encode_context(dec.device_memory(mem), ctx_len, forced)
        lp = dec.teacher_forward(subs)[0] if dtype == "bf16" else np.zeros(1)
        dec.run()
        return [lp, dec.get_logits()[0], dec.collect()["tokens"]]
    want = results()

    def shifted(t):
        buf = torch.empty(t.numel() + 1, dtype=t.dtype, device=t.device)
        buf[1:] = t.reshape(-1)
        return buf
    tables = ["embed", "final_norm"] + [f"l{l}.norm{k}" for l in range(wl.n_layers) for k in (1, 2, 3)]
    keep = {k: shifted(dec._w[k]) for k in tables}
    at = {k: t.data_ptr() + t.element_size() for k, t in keep.items()}
    for l in range(wl.n_layers):
        for j, name in enumerate(B.LAYER_TENSORS):
            dec._layer_ptrs[l * len(B.LAYER_TENSORS) + j] = at.get(f"l{l}.{name}", dec._w[f"l{l}.{name}"].data_ptr())
    w = B.PdWeights()
    w.embed, w.final_norm, w.lm_head, w.rel_bias = at["embed"], at["final_norm"], dec._w["lm_head"].data_ptr(), None
    w.layer = C.cast(dec._layer_ptrs, C.POINTER(C.c_void_p))
    torch.cuda.synchronize()
    B._lib.pd_destroy(dec._h)
    dec._h = B._H()
    st = B._lib.pd_init(C.byref(dec.cfg), C.byref(w), C.c_void_p((dec._ws.data_ptr() + 255) // 256 * 256), C.c_size_t(dec.workspace_bytes),
                        C.c_void_p(dec.stream.cuda_stream), C.byref(dec._h))
    assert st == 0
    for a, b in zip(want, results()):
        assert np.array_equal(a, b)
    dec.close()


@pytest.mark.parametrize("dtype,batch,rows", [("fp32", 16384, 49), ("fp32", 40000, 17), ("bf16", 22000, 33), ("bf16", 65535, 2)])
def test_cross_attention_of_many_sequences(dtype, batch, rows):
    """More sequences than a grid dimension holds chunks of rows.  The first, a middle and the last sequence against fp64; tolerances as
    for the operator's other tests (fp32 sums of 8 keys; bf16: weights and result rounded, 2^-9 each)."""
    import torch
    from paper_2506_23431_b200 import binding as B
    dev, td = torch.device("cuda", 0), torch.float32 if dtype == "fp32" else torch.bfloat16
    gen = torch.Generator(device=dev)
    gen.manual_seed(batch)
    q = torch.randn(batch, rows, 64, generator=gen, device=dev).to(td)
    kv = torch.randn(batch, 1, 2, 8, 64, generator=gen, device=dev).to(td)
    n_rows = torch.full((batch,), rows, dtype=torch.int32, device=dev)
    ctx_len = torch.full((batch,), 7, dtype=torch.int32, device=dev)
    out = B.cross_attention(q, kv, n_rows, ctx_len, 0.125, 1)
    for b in (0, batch // 2, batch - 1):
        w = torch.softmax(0.125 * q[b].double() @ kv[b, 0, 0, :7].double().T, -1)
        ref = w @ kv[b, 0, 1, :7].double()
        assert (out[b].double() - ref).abs().max().item() <= (2e-5 if dtype == "fp32" else 2 * 2.0 ** -9 * kv[b].abs().max().item())


@pytest.mark.parametrize("dtype,rows", [("fp32", 4), ("bf16", 4), ("bf16", 40)])
@pytest.mark.parametrize("first,last", [(0, 32), (32, 64), (96, 97), (256, 300)])
def test_cross_attention_with_keys_out_of_range(dtype, rows, first, last):
    """Keys that are no numbers make the head's rows none, wherever their tile falls; keys whose scores overflow to -inf weigh nothing.  The
    other head is not touched.  Both attention kernels, one split and three; tolerance as for the operator's other tests."""
    import torch
    from paper_2506_23431_b200 import binding as B
    dev, td = torch.device("cuda", 0), torch.float32 if dtype == "fp32" else torch.bfloat16
    gen = torch.Generator(device=dev)
    gen.manual_seed(first)
    q = (0.5 + torch.rand(1, rows, 128, generator=gen, device=dev)).to(td)
    kv = torch.randn(1, 2, 2, 300, 64, generator=gen, device=dev).to(td)
    n_rows = torch.full((1,), rows, dtype=torch.int32, device=dev)
    ctx_len = torch.full((1,), 300, dtype=torch.int32, device=dev)
    for splits in (1, 3):
        for bad in (float("nan"), -3e38):
            keys = kv.clone()
            keys[0, 1, 0, first:last] = bad
            out = B.cross_attention(q, keys, n_rows, ctx_len, 0.125, splits)[0].double()
            for h in (0, 1):
                got = out[:, 64 * h:64 * h + 64]
                if h == 1 and bad != bad:
                    assert torch.isnan(got).all()
                    continue
                s = 0.125 * q[0, :, 64 * h:64 * h + 64].double() @ kv[0, h, 0].double().T
                if h == 1:
                    s[:, first:last] = -float("inf")
                ref = torch.softmax(s, -1) @ kv[0, h, 1].double()
                assert (got - ref).abs().max().item() <= (2e-5 if dtype == "fp32" else 2 * 2.0 ** -9 * kv.abs().max().item())


@pytest.mark.parametrize("vocab", [301, 2304])
@pytest.mark.parametrize("first", [0, 4, 297])
def test_log_probabilities_of_logits_out_of_range(vocab, first):
    """Four output vectors that are no numbers (a thread's first load of a row among them) leave no row a log-probability; four whose logits
    overflow to -inf take no part in the sums: the row's log-probability is that of the other words."""
    from paper_2506_23431_b200.binding import PipelinedDecoder
    wl = W.CONFIGS["bart_base"].scaled(name="tf_nan", n_layers=1, d_model=128, n_heads=2, d_ff=256, vocab=vocab, norm_gain_std=0.1, batch=1, ctx=40,
                                       sub_max=2, delta_t=2, max_sub_len=15, length_dist=("uniform", 5, 15), time_max=25, pos_mode=ROPE)
    weights = W.make_weights(wl)
    # the embedding's first column dominates and the final norm keeps nothing else: every hidden state is +c, 0, 0, ...
    weights["embed"][:, 0] = 64.0
    weights["final_norm"][:] = 0
    weights["final_norm"][0] = 1
    subs = [[[20, 21, 22], [23]]]
    lp = {}
    for bad in (0.0, np.nan, -3e38):
        w = dict(weights, lm_head=weights["lm_head"].copy())
        w["lm_head"][first:first + 4, 0] = bad
        w["lm_head"][wl.sep_id, 0] = weights["lm_head"][wl.sep_id, 0]
        dec = PipelinedDecoder(wl.hyper(), w, wl.batch)
        dec.encode_context(dec.device_memory(W.make_encoder_memory(wl)), [wl.ctx], None)
        lp[str(bad)], _, logits = dec.teacher_forward(subs, want_logits=True)
        z = logits.cpu().numpy().astype(np.float64)
        tgt = [20, 21, 22, wl.sep_id, 23, wl.sep_id]
        if bad == bad:
            keep = np.isfinite(z)
            assert (~keep).sum() == (0 if bad == 0 else 6 * (4 - (first <= wl.sep_id < first + 4)))
            want = [z[r, t] - np.log(np.exp(z[r][keep[r]] - z[r][keep[r]].max()).sum()) - z[r][keep[r]].max() for r, t in enumerate(tgt)]
            assert np.abs(lp[str(bad)] - want).max() <= 1e-4
        else:
            assert np.isnan(lp[str(bad)]).all()
        dec.close()


@pytest.mark.parametrize("ctx,bad", [(130, (0, 64)), (130, (0, 128)), (300, (64, 200)), (64, (0, 63))])
def test_teacher_forward_with_keys_whose_scores_overflow(ctx, bad):
    """Keys that score -inf with every query - a row's whole first half tile among them - weigh nothing: the forward over a context that
    holds them equals the oracle's over the rest (cross-attention has no positions)."""
    from oracle import pipelined_decoder as O
    from paper_2506_23431_b200.binding import PipelinedDecoder
    wl = W.CONFIGS["bart_base"].scaled(name="tf_over", n_layers=1, d_model=128, n_heads=2, d_ff=256, vocab=301, norm_gain_std=0.1, batch=1, ctx=ctx,
                                       sub_max=5, delta_t=2, max_sub_len=15, length_dist=("uniform", 10, 15), time_max=25, pos_mode=ROPE)
    weights, mem, subs = W.make_weights(wl), W.make_encoder_memory(wl), [[[5, 6, 7, 8], [9, 10], [11] * 15, [12] * 15, [13] * 15]]
    # every query is positive (the first column of every state dominates and feeds all of wq_c's columns), the bad positions' keys
    # are -2e38 in every column; values take nothing from the column that makes them so
    weights["embed"][:, 0] = 8.0
    weights["l0.wq_c"][0] = 0.5
    weights["l0.wkv_c"][0, :128], weights["l0.wkv_c"][0, 128:] = 1.0, 0.0
    mem[0, :, 0] = 0
    weights = {k: W.bf16_round(v) if k != "rel_bias" else v for k, v in weights.items()}
    worse = mem.copy()
    worse[0, bad[0]:bad[1], 0] = -2e38
    keep = np.ones(ctx, bool)
    keep[bad[0]:bad[1]] = False
    dec = PipelinedDecoder(wl.hyper(), weights, wl.batch)
    dec.encode_context(dec.device_memory(W.bf16_round(worse)), [ctx], None)
    got = dec.teacher_forward(subs, want_logits=True)[2].cpu().numpy()
    ref = O.PipelinedDecoderOracle(weights, wl.hyper()).teacher_forward(mem[0][keep], int(keep.sum()), subs[0])["logits"]
    assert np.abs(got - ref).max() <= 2e-2
    dec.close()


@pytest.mark.parametrize("dtype,rows", [("fp32", 1), ("fp32", 17), ("bf16", 33)])
@pytest.mark.parametrize("ctx,splits", [(1, 1), (32, 4), (33, 1), (257, 2), (300, 4), (515, 3)])
def test_plain_alu_attention_with_few_tiles_per_cta(dtype, rows, ctx, splits):
    """More (sequence, head, chunk) triples than SMs, so that a CTA has as many warps as it has tiles for: one to eight, with ragged contexts
    and rows, one split and several; tolerances as for the operator's other tests."""
    import torch
    from paper_2506_23431_b200 import binding as B
    q, kv, n_rows, ctx_len = cross_case(ctx, 40, rows, 4, ctx, dtype)
    ref = oracle_cross(q, kv, n_rows, ctx_len, 4, 0.125)
    dev, td = torch.device("cuda", 0), torch.float32 if dtype == "fp32" else torch.bfloat16
    out = B.cross_attention(torch.from_numpy(q).to(dev, td), torch.from_numpy(kv).to(dev, td), torch.from_numpy(n_rows).to(dev),
                            torch.from_numpy(ctx_len).to(dev), 0.125, splits)
    tol = 2e-5 if dtype == "fp32" else 2 * 2.0 ** -9 * max(1.0, np.abs(kv[np.isfinite(kv)]).max())
    assert np.abs(out.float().cpu().numpy().astype(np.float64) - ref).max() <= tol


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("which", ["self_attn", "cross_attn"])
def test_timed_attention_launches_do_not_overlap(dtype, which):
    """pd_time_attention reports the duration of a launch, so none may begin under the one before (as they do inside a step)."""
    import torch
    from torch.profiler import ProfilerActivity, profile
    from paper_2506_23431_b200.binding import PipelinedDecoder
    wl = W.CONFIGS["bart_base" if dtype == "bf16" else "tiny"].scaled(name="timed", batch=2, ctx=700, n_layers=4, sub_max=6, vocab=500)
    dec = PipelinedDecoder(wl.hyper(), W.make_weights(wl), wl.batch)
    dec.encode_context(dec.device_memory(W.make_encoder_memory(wl)), W.make_ctx_len(wl), W.make_forced_len(wl))
    for _ in range(4):
        dec.step()
    dec.time_attention(which, 1)
    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        assert dec.time_attention(which, 5) > 0
    spans = sorted((e.time_range.start, e.time_range.end) for e in prof.events() if "attn" in e.name)
    dec.close()
    if not spans:
        pytest.skip("the profiler records no kernels here")
    assert len(spans) >= 6 * wl.n_layers
    assert all(b[0] >= a[1] for a, b in zip(spans, spans[1:]))


@pytest.mark.parametrize("kv8", [True, False])
@pytest.mark.parametrize("batch,heads,ctx", [(16, 12, 1024), (16, 16, 512), (8, 12, 2048), (2, 4, 96)])
def test_decodes_of_few_rows_repeat_bit_for_bit(batch, heads, ctx, kv8):
    """The packed path, whose launches overlap: residual stream and tokens of a whole decode, again and again, on one handle."""
    from paper_2506_23431_b200 import binding as B
    wl = W.CONFIGS["bart_base"].scaled(name="repeat", batch=batch, n_layers=4, d_model=64 * heads, n_heads=heads, d_ff=256 * heads, vocab=2000, ctx=ctx,
                                       sub_max=8, delta_t=4, max_sub_len=24, length_dist=("uniform", 10, 24), time_max=40, pos_mode=T5,
                                       kv_c_dtype="e4m3" if kv8 else "same")
    dec = B.PipelinedDecoder(wl.hyper(), W.make_weights(wl), wl.batch)
    mem, ctx_len, forced = dec.device_memory(W.make_encoder_memory(wl)), W.make_ctx_len(wl), W.make_forced_len(wl)
    first = None
    for _ in range(12):
        dec.encode_context(mem, ctx_len, forced)
        for _ in range(36):
            dec.step()
        rows = dec.batch * dec.rows_per_seq
        got = (dec.debug_read(B.PD_BUF_X, np.float32, rows * wl.d_model).copy(), dec.get_chosen().copy())
        first = first or got
        assert np.array_equal(got[0], first[0]) and np.array_equal(got[1], first[1])
    dec.close()


PACKED = [
    # sequences, open rows per sequence, inner width, positions, longest subsequence, 8-bit context
    (5, 26, 64, ROPE, 28, False),       # 130 rows allocated, register products beyond 128; an inner width of one block
    (19, 31, 1088, T5, 33, True),       # 589 rows: register products still; a reduction over two CTAs
    (18, 32, 2112, ROPE, 34, False),    # 576 rows: the inner products on tensor memory; a reduction over three pairs of CTAs
    (24, 32, 4160, T5, 36, False),      # 768 rows, the most that run packed; four pairs, the last one shorter
    (25, 31, 192, T5, 33, False),       # 775 rows: the kernels beyond
    (90, 7, 256, ROPE, 40, False),      # 630 rows, two pages per subsequence
]


@pytest.mark.parametrize("batch,rows,d_ff,pos,length,kv8", PACKED)
def test_decode_on_tensor_memory_products(batch, rows, d_ff, pos, length, kv8):
    """More rows than the register products take: rows of 1 to all of a group, widths that end inside a slice of columns (192, 576)."""
    wl = W.CONFIGS["bart_base"].scaled(name="packed", batch=batch, sub_max=rows, d_ff=d_ff, pos_mode=pos, max_sub_len=length, time_max=min(rows + 6, 96),
                                       length_dist=("uniform", max(1, length - 4), length), kv_c_dtype="e4m3" if kv8 else "same",
                                       **dict(BASE, ctx=144 if kv8 else 150))
    s = check(wl, rows=[0, batch - 1], ragged=True, free_run=False)
    assert s["max_err"] < parity.TOL["bf16"]


WHOLE = [
    # sequences, open rows per sequence, heads, inner width, positions, 8-bit context; weights and rows that put every product on tensor memory
    (18, 32, 9, 1088, ROPE, False),     # 576 rows of width 576, which ends inside a pair's columns; a reduction over two pairs, the second one block shorter
    (18, 32, 9, 1088, T5, True),
    (8, 26, 16, 2112, ROPE, False),     # 208 rows of width 1024, the longest reduction that is not split; an inner one over three pairs
    (8, 27, 16, 4160, T5, False),       # 216 rows; four pairs
]


@pytest.mark.parametrize("batch,rows,heads,d_ff,pos,kv8", WHOLE)
def test_decode_with_every_product_on_tensor_memory(batch, rows, heads, d_ff, pos, kv8):
    wl = W.CONFIGS["bart_base"].scaled(name="whole", batch=batch, sub_max=rows, d_ff=d_ff, pos_mode=pos, max_sub_len=rows + 2, time_max=rows + 6,
                                       length_dist=("uniform", rows - 4, rows + 2), kv_c_dtype="e4m3" if kv8 else "same",
                                       **dict(BASE, d_model=64 * heads, n_heads=heads, ctx=48))
    s = check(wl, rows=[0, batch - 1], ragged=True, free_run=False)
    assert s["max_err"] < parity.TOL["bf16"]


RULES = [
    # sequences, open rows per sequence, heads, inner width -> products
    (10, 30, 1, 4800),     # 300 rows: register products that take three batches of rows in one row group
    (10, 31, 1, 4800),     # 310 rows: the wide ones on tensor memory, the others on registers
    (24, 32, 4, 1024),     # 768 rows: the inner products on tensor memory, the others on registers
    (7, 30, 17, 192),      # 210 rows of width 1088: the most that run packed beyond width 1024 (211)
    (8, 27, 17, 192),      # 216 rows: the library's
]


@pytest.mark.parametrize("batch,rows,heads,d_ff", RULES)
def test_decode_where_the_products_change_kernels(batch, rows, heads, d_ff):
    wl = W.CONFIGS["bart_base"].scaled(name="rules", batch=batch, sub_max=rows, d_ff=d_ff, pos_mode=ROPE, max_sub_len=rows + 2, time_max=rows + 6,
                                       length_dist=("uniform", rows - 4, rows + 2), **dict(BASE, d_model=64 * heads, n_heads=heads, ctx=40))
    s = check(wl, rows=[0, batch - 1], ragged=True, free_run=False)
    assert s["max_err"] < parity.TOL["bf16"]


@pytest.mark.parametrize("pos", [ROPE, T5])
@pytest.mark.parametrize("heads", [17, 33, 49])
def test_decode_on_split_tensor_memory_products(heads, pos):
    """Widths whose every product is split over two, three and four pairs, the rows of a group (5 to 130) in all its sizes.  In rotary mode
    the pairs ask for the positions of whole chunks of rows, of rows beyond the group's too.  A logit is a product of a normalised row, whose length
    is sqrt(width), with a row of lm_head: at one weight scale its error grows with sqrt(width) (2.4e-2 at 2112).  The weights shrink by that factor, so that
    logits and errors have the scale that the bar is for, that of width 1024."""
    wl = W.CONFIGS["bart_base"].scaled(name="split", batch=5, sub_max=26, d_ff=192, pos_mode=pos, max_sub_len=28, time_max=32,
                                       length_dist=("uniform", 24, 28), **dict(BASE, d_model=64 * heads, n_heads=heads, n_layers=1, ctx=40,
                                                                            weight_std=0.02 * (1024 / (64 * heads)) ** 0.5))
    s = check(wl, rows=[0, 4], ragged=True, free_run=False)
    assert s["max_err"] < parity.TOL["bf16"]


@pytest.mark.parametrize("kv8", [True, False])
@pytest.mark.parametrize("batch,heads,ctx", [(24, 16, 512), (40, 12, 300)])
def test_decodes_of_many_packed_rows_repeat_bit_for_bit(batch, heads, ctx, kv8):
    test_decodes_of_few_rows_repeat_bit_for_bit(batch, heads, ctx // 16 * 16, kv8)


def test_two_handles_side_by_side_on_tensor_memory_products():
    """Steps of two handles on streams of their own, whose pairs of CTAs share SMs and tensor memory: each gives what it gives alone."""
    from paper_2506_23431_b200 import binding as B
    runs = []
    for batch, heads in ((24, 16), (40, 12)):
        wl = W.CONFIGS["bart_base"].scaled(name="beside", batch=batch, n_layers=3, d_model=64 * heads, n_heads=heads, d_ff=256 * heads, vocab=2000, ctx=300,
                                           sub_max=8, delta_t=4, max_sub_len=24, length_dist=("uniform", 10, 24), time_max=40, pos_mode=T5)
        dec = B.PipelinedDecoder(wl.hyper(), W.make_weights(wl), wl.batch)
        runs.append((dec, (dec.device_memory(W.make_encoder_memory(wl)), W.make_ctx_len(wl), W.make_forced_len(wl)), batch * dec.rows_per_seq * wl.d_model))

    def result(dec, n):
        return dec.debug_read(B.PD_BUF_X, np.float32, n).copy(), dec.get_chosen().copy()

    alone = []
    for dec, args, n in runs:
        dec.encode_context(*args)
        for _ in range(30):
            dec.step()
        alone.append(result(dec, n))
    for _ in range(4):
        for dec, args, _n in runs:
            dec.encode_context(*args)
        for _ in range(30):
            for dec, _args, _n in runs:
                dec.step()
        for (dec, _args, n), want in zip(runs, alone):
            got = result(dec, n)
            assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
    for dec, _args, _n in runs:
        dec.close()


@pytest.mark.parametrize("batch,rows", [(15, 3), (16, 3), (16, 20), (49, 3), (50, 3), (98, 3), (99, 3), (148, 3), (149, 3)])
def test_decode_where_8_bit_launches_change_their_spread(batch, rows):
    """45, 48, 147, 150, 294, 297, 444 and 447 segments over 8-bit context: launches behind the kernel before, and under it with one to four CTAs per SM
    (20 rows per sequence: the form of two row tiles)."""
    wl = W.CONFIGS["bart_base"].scaled(name="spread", batch=batch, sub_max=rows, d_ff=192, pos_mode=T5, max_sub_len=rows + 3, time_max=rows + 6,
                                       length_dist=("uniform", 2, rows + 3), kv_c_dtype="e4m3", **dict(BASE, n_layers=1, ctx=272))
    s = check(wl, rows=[0, batch - 1], ragged=True, free_run=False)
    assert s["max_err"] < parity.TOL["bf16"]

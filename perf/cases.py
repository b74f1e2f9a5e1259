"""The workloads by which this library's speed is judged, through its public entry points.

A serving program does four kinds of work with the library: it prepares weights once (the quantisers), it runs the
verification pass of a speculative-decoding step again and again (tiny and full models, one sequence or a batch, chains and
trees, blocks of one row up to the 64-row chunks that fill a cache from a prompt; int8, W8A8 and bf16 verifiers), it drafts
and samples around that pass, and it calls single linear layers from code of its own.  Model sizes are the ones of
`paper_2603_01399_b200.synth`.
"""
from __future__ import annotations

import math
import random

import torch

from paper_2603_01399_b200 import binding as Q
from paper_2603_01399_b200 import synth

DEV = "cuda"


def listed():
    return [
        # A very small decoder, called without a plan: launches and host work are all there is.
        {"name": "tiny_chain", "op": "verify", "model": "tiny", "weights": "int8", "batch": 1, "rows": 5, "tree": False,
         "prefix_min": 64, "prefix_max": 64, "ragged": False, "logits": True, "entry": "call", "commit": False,
         "in_place": False},
        # The headline: one user, a 5-token draft on a 1024-token context, the pass frozen as a plan.
        {"name": "chain_8b", "op": "verify", "model": "qwen3_8b", "weights": "int8", "batch": 1, "rows": 6, "tree": False,
         "prefix_min": 1024, "prefix_max": 1024, "ragged": False, "logits": True, "entry": "plan", "commit": False,
         "in_place": False},
        # A serving step: eight users with contexts of very different length, host buffers in and out.
        {"name": "batch8_8b", "op": "verify", "model": "qwen3_8b", "weights": "int8", "batch": 8, "rows": 9, "tree": False,
         "prefix_min": 512, "prefix_max": 4096, "ragged": False, "logits": True, "entry": "host", "commit": False,
         "in_place": False},
        # Tree drafts (16 candidates and the root) on the larger model, with the commit that follows the pass.
        {"name": "tree_14b", "op": "verify", "model": "qwen3_14b", "weights": "int8", "batch": 4, "rows": 17, "tree": True,
         "prefix_min": 2048, "prefix_max": 2048, "ragged": False, "logits": True, "entry": "plan", "commit": True,
         "in_place": False},
        # Prompts entering the cache: one 64-row chunk of each of eight sequences, the last chunks ragged, no logits wanted.
        {"name": "prefill_8b", "op": "verify", "model": "qwen3_8b", "weights": "int8", "batch": 8, "rows": 64, "tree": False,
         "prefix_min": 0, "prefix_max": 1024, "ragged": True, "logits": False, "entry": "call", "commit": True,
         "in_place": False},
        # The paper's own arithmetic (int8 activations too), the headline's shape.
        {"name": "w8a8_8b", "op": "verify", "model": "qwen3_8b", "weights": "w8a8", "batch": 1, "rows": 6, "tree": False,
         "prefix_min": 1024, "prefix_max": 1024, "ragged": False, "logits": True, "entry": "plan", "commit": False,
         "in_place": False},
        # The unquantised verifier that the paper compares with, the headline's shape.
        {"name": "bf16_8b", "op": "verify", "model": "qwen3_8b", "weights": "bf16", "batch": 1, "rows": 6, "tree": False,
         "prefix_min": 1024, "prefix_max": 1024, "ragged": False, "logits": True, "entry": "plan", "commit": False,
         "in_place": False},
        # One small linear layer called from a program of its own: an output projection with its residual.
        {"name": "linear_o", "op": "linear", "weights": "int8", "m": 5, "n": 4096, "k": 4096, "f32": False, "residual": True,
         "static": False},
        # The W8A8 linear layer on a batch: a gate+up projection.
        {"name": "linear_w8a8_gateup", "op": "w8a8", "m": 40, "n": 24576, "k": 4096, "f32": False, "residual": False,
         "smooth": True},
        # 4-bit weights: a down projection with its residual.
        {"name": "linear_w4_down", "op": "w4", "m": 16, "n": 4096, "k": 12288, "f32": False, "residual": True},
        # Offline weight preparation: the largest matrix of a layer.
        {"name": "quantize_gateup", "op": "quantize", "kind": "int8", "n": 24576, "k": 4096},
        # Around the pass in a sampling server: prompt-lookup drafts and the stochastic acceptance of the last block.
        {"name": "draft_and_sample", "op": "sample", "batch": 8, "rows": 9, "vocab": 151936, "history": 4096,
         "with_q": True},
    ]


def _log(rng, lo, hi):
    """A whole number between lo and hi, spread over the logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))


def _matrix_size(rng):
    """(n, k) of a linear layer: one of a named model's, or any in their range (k a multiple of 16)."""
    if rng.random() < 0.6:
        shape = synth.SHAPES[rng.choice(["qwen3_8b", "qwen3_14b", "tiny"])]
        _, n, k = rng.choice(shape.linear_shapes())
        return n, k
    return _log(rng, 200, 40000), 16 * _log(rng, 16, 1088)


def draw(rng: random.Random):
    op = rng.choice(["verify"] * 5 + ["linear"] * 3 + ["w8a8", "w4", "quantize", "sample"])
    if op == "verify":
        model = rng.choice(["tiny", "tiny_qknorm", "qwen3_8b", "qwen3_8b", "qwen3_8b", "qwen3_14b"])
        weights = rng.choice(["int8", "int8", "int8", "w8a8", "bf16"])
        if model == "qwen3_14b" and weights == "bf16":
            weights = "int8"
        tree = rng.random() < 0.25
        rows = rng.choice([17, 29]) if tree else rng.choice([_log(rng, 1, 10), _log(rng, 1, 64)])
        batch = _log(rng, 1, 8)
        # no more than the largest listed case: rows of the whole block by the size of the model
        most = {"qwen3_14b": 128, "qwen3_8b": 384}.get(model, 512) if weights != "bf16" else 144
        batch = max(1, min(batch, most // rows))
        hi = _log(rng, 16, 4096) if batch <= 4 else _log(rng, 16, 2048)
        lo = max(0, int(hi * rng.choice([1.0, rng.random()])))
        fits = batch * rows <= 8 and weights == "int8"
        return {"op": "verify", "model": model, "weights": weights, "batch": batch, "rows": rows, "tree": tree,
                "prefix_min": lo, "prefix_max": hi, "ragged": False, "logits": rng.random() < 0.8,
                "entry": rng.choice(["call", "plan", "plan", "host"]), "commit": rng.random() < 0.4,
                "in_place": bool(fits and rng.random() < 0.25)}
    if op == "linear":
        n, k = _matrix_size(rng)
        m = _log(rng, 1, 64) if rng.random() < 0.7 else _log(rng, 1, 512)
        f32 = n > 100000 or rng.random() < 0.3
        static = m <= 8 and n <= 6144 and rng.random() < 0.3
        return {"op": "linear", "weights": rng.choice(["int8", "int8", "bf16"]), "m": m, "n": n, "k": k, "f32": f32,
                "residual": bool(not f32 and rng.random() < 0.4), "static": bool(static)}
    if op == "w8a8":
        n, k = _matrix_size(rng)
        f32 = n > 100000 or rng.random() < 0.3
        return {"op": "w8a8", "m": _log(rng, 1, 128), "n": n, "k": k, "f32": f32,
                "residual": bool(not f32 and rng.random() < 0.4), "smooth": rng.random() < 0.7}
    if op == "w4":
        n, k = _matrix_size(rng)
        f32 = n > 100000 or rng.random() < 0.3
        return {"op": "w4", "m": _log(rng, 1, 64), "n": n, "k": max(256, k // 128 * 128), "f32": f32,
                "residual": bool(not f32 and rng.random() < 0.4)}
    if op == "quantize":
        n, k = _matrix_size(rng)
        kind = rng.choice(["int8", "smoothed", "int4", "activations"])
        return {"op": "quantize", "kind": kind, "n": _log(rng, 1, 512) if kind == "activations" else n,
                "k": max(256, k // 128 * 128)}
    return {"op": "sample", "batch": _log(rng, 1, 16), "rows": _log(rng, 2, 10), "vocab": _log(rng, 1024, 151936),
            "history": _log(rng, 64, 16384), "with_q": rng.random() < 0.5}


# ---- sizes that follow from a case ----------------------------------------------------------------------------------
def _prefixes(case):
    """The sequences' cached lengths, spread evenly over the case's range."""
    lo, hi, b = case["prefix_min"], case["prefix_max"], case["batch"]
    return [lo + (hi - lo) * i // max(1, b - 1) for i in range(b)]


def _block_lens(case):
    """Rows of each sequence's block: all of them, or ragged (a prompt's last chunk, a drafter that found less)."""
    t = case["rows"]
    return [max(1, t - (7 * i) % max(1, t // 2 + 1)) if case["ragged"] else t for i in range(case["batch"])]


def _parents(case):
    return synth.tree_parents_16() if case["rows"] == 17 else synth.tree_parents_full()


# ---- inputs ---------------------------------------------------------------------------------------------------------
def _gen(seed, what, layer=0):
    g = torch.Generator(device=DEV)
    g.manual_seed((seed * 1_000_003 + sum(ord(c) * 131 ** i for i, c in enumerate(what)) + 7919 * layer) % (2 ** 62))
    return g


def _normal(dims, std, g, dtype=torch.bfloat16):
    return torch.empty(dims, dtype=dtype, device=DEV).normal_(0.0, std, generator=g)


def _uniform(dims, lo, hi, g, dtype=torch.float32):
    return torch.empty(dims, dtype=dtype, device=DEV).uniform_(lo, hi, generator=g)


def _model(case, seed, max_seq):
    """A decoder of the named sizes with seeded weights, and the token it predicts after each token.

    Random weights alone give flat predictions, in which the last bit of a sum decides the top choice; a trained verifier
    is sure of most of its tokens.  So each token has a successor, whose LM-head row leans towards that token's embedding,
    and the projections back into the residual stream are scaled by 1/sqrt(2 layers)."""
    shape = synth.SHAPES[case["model"]]
    host = torch.Generator()
    host.manual_seed(seed * 7 + 3)
    successor = torch.randperm(shape.vocab, generator=host)
    embed = _normal((shape.vocab, shape.hidden), 1.0, _gen(seed, "embed"))
    dims = {name: (n, k) for name, n, k in shape.linear_shapes()}
    back = 0.02 / math.sqrt(2 * shape.n_layers)

    def master(kind, layer):
        g = _gen(seed, kind, layer)
        if kind == "embed":
            return embed
        if kind in ("q_norm", "k_norm"):
            return _uniform((shape.head_dim,), 0.5, 1.5, g, torch.bfloat16)
        if kind.endswith("norm"):
            return _uniform((shape.hidden,), 0.5, 1.5, g, torch.bfloat16)
        w = _normal(dims[kind], back if kind in ("o", "down") else 0.02, g)
        if kind == "lm_head":
            w[successor.to(DEV)] += embed * (40.0 / shape.hidden)
        return w

    model = Q.Model.from_master(
        shape, master, max_seq, int8=case["weights"] != "bf16", device=DEV, act_int8=case["weights"] == "w8a8",
        get_act_absmax=lambda kind, layer: synth.activation_absmax(shape, kind, layer, seed, DEV),
        weights_in_place=case["in_place"])
    return model, successor.tolist()


def _draft_tokens(case, vocab, successor, rng):
    """Blocks as drafters make them: the last emitted token, then guesses, 3 in 10 of them wrong; in a tree one child
    of a node is the good guess and the others are random."""
    out = []
    for _ in range(case["batch"]):
        row = [rng.randrange(vocab)]
        parents = _parents(case) if case["tree"] else synth.chain_parents(case["rows"])
        guessed = set()
        for p in parents[1:]:
            good = p not in guessed and rng.random() < 0.7
            guessed.add(p)
            row.append(successor[row[p]] if good else rng.randrange(vocab))
        out.append(row)
    return torch.tensor(out, dtype=torch.int32)


def _prepare_verify(case, seed):
    b, t = case["batch"], case["rows"]
    max_seq = (case["prefix_max"] + t + 63) // 64 * 64
    model, successor = _model(case, seed, max_seq)
    shape = model.shape
    dims = (shape.n_layers, b, shape.n_kv_heads, max_seq, shape.head_dim)
    lens = torch.tensor(_prefixes(case), dtype=torch.int32, device=DEV)
    kv = Q.KVCache(shape, b, max_seq, DEV, k=_normal(dims, 1.0, _gen(seed, "kv_k")), v=_normal(dims, 1.0, _gen(seed, "kv_v")),
                   seq_len=lens.clone())
    buf = Q.VerifyBuffers(model, b, t, want_logits=case["logits"], tree=case["tree"], device=DEV)
    tokens = _draft_tokens(case, shape.vocab, successor, random.Random(seed))
    buf.tokens.copy_(tokens)
    buf.block_len.copy_(torch.tensor(_block_lens(case), dtype=torch.int32))
    if case["tree"]:
        buf.parents.copy_(torch.tensor([_parents(case)] * b, dtype=torch.int32))
    s = {"case": case, "model": model, "kv": kv, "buf": buf, "lens": lens, "plan": None}
    if case["commit"] and not case["tree"] and not case["logits"]:
        s["whole"] = buf.block_len - 1      # a prompt's chunk: every row stays
    if case["entry"] != "call":
        s["plan"] = Q.Plan(model, kv, buf)
    if case["entry"] == "host":
        pin = lambda x: x.cpu().pin_memory()  # noqa: E731
        s["host"] = {"tokens": tokens.pin_memory(), "accept_len": pin(buf.accept_len), "bonus": pin(buf.bonus),
                     "block_len": pin(buf.block_len), "path": pin(buf.accept_path), "status": pin(buf.status[:1]),
                     "parents": pin(buf.parents) if case["tree"] else None}
    return s


def _prepare_linear(case, seed):
    m, n, k = case["m"], case["n"], case["k"]
    s = {"case": case, "x": _normal((m, k), 1.0, _gen(seed, "x"))}
    w = _normal((n, k), 0.02, _gen(seed, "w"))
    s["res"] = _normal((m, n), 1.0, _gen(seed, "res")) if case["residual"] else None
    s["smooth"] = s["delta"] = None
    if case["op"] == "w4":
        s["w"], s["delta"] = Q.quasar_quantize_int4(w)
    elif case["op"] == "w8a8":
        if case["smooth"]:
            peak = _uniform((k,), 0.5, 4.0, _gen(seed, "peak"))
            outlier = _uniform((k,), 0.0, 1.0, _gen(seed, "outlier")) < 0.01
            peak = torch.where(outlier, peak * 20, peak)
            s["x"] = (s["x"].float() * (peak / 4)).to(torch.bfloat16)
            s["smooth"] = Q.quasar_smoothing_factors(peak, w)
        s["w"], s["delta"] = Q.quasar_quantize_weights_smoothed(w, s["smooth"])
    elif case["weights"] == "int8":
        s["w"], s["delta"] = Q.quasar_quantize(w)
    else:
        s["w"] = w
    if case["op"] == "linear":
        s["out"] = torch.empty((m, n), dtype=torch.float32 if case["f32"] else torch.bfloat16, device=DEV)
        if not case["static"]:
            s["workspace"] = torch.zeros(Q.quasar_linear_workspace_bytes(m, n, k), dtype=torch.uint8, device=DEV)
    return s


def _prepare_sample(case, seed):
    b, t, v = case["batch"], case["rows"], case["vocab"]
    # The logits of a trained model: nearly all of the probability on a few dozen tokens of each row.
    logits = _normal((b, t, v), 1.3, _gen(seed, "logits"), torch.float32)
    likely = torch.randint(0, v, (b, t, 32), generator=_gen(seed, "likely"), device=DEV)
    logits.scatter_(2, likely, _uniform((b, t, 32), 16.0, 20.0, _gen(seed, "height")))
    q = None
    if case["with_q"]:      # the drafter's distribution: near the verifier's
        q = torch.softmax(logits + _normal((b, t, v), 0.5, _gen(seed, "q"), torch.float32), dim=-1)
    tokens = torch.zeros((b, t), dtype=torch.int32, device=DEV)
    tokens[:, 1:] = likely[:, :-1, 0].to(torch.int32)       # draft i+1 is one of the likely tokens after row i
    # Histories with repeats, as prompts have: phrases of a few tokens from a small stock, cut at different lengths.
    rng = random.Random(seed)
    phrases = [[rng.randrange(v) for _ in range(rng.randrange(3, 12))] for _ in range(40)]
    hist, lens = torch.zeros((b, case["history"]), dtype=torch.int32), []
    for i in range(b):
        row = []
        while len(row) < case["history"]:
            row += rng.choice(phrases) if rng.random() < 0.5 else [rng.randrange(v) for _ in range(6)]
        lens.append(max(8, case["history"] - (i * case["history"]) // (2 * b)))
        cut = row[:lens[-1]]
        tail = rng.choice(phrases)[:3]
        cut[-3:] = tail                                     # the text ends inside a phrase seen before
        hist[i, :len(cut)] = torch.tensor(cut, dtype=torch.int32)
    return {"case": case, "logits": logits, "q": q, "tokens": tokens, "history": hist.to(DEV),
            "hist_len": torch.tensor(lens, dtype=torch.int32, device=DEV),
            "block_len": torch.full((b,), t, dtype=torch.int32, device=DEV),
            "r_accept": _uniform((b, t), 0.0, 1.0, _gen(seed, "ra")), "r_sample": _uniform((b,), 0.0, 1.0, _gen(seed, "rs"))}


def prepare(case, seed):
    if case["op"] == "verify":
        return _prepare_verify(case, seed)
    if case["op"] in ("linear", "w8a8", "w4"):
        return _prepare_linear(case, seed)
    if case["op"] == "sample":
        return _prepare_sample(case, seed)
    s = {"case": case, "w": _normal((case["n"], case["k"]), 1.0 if case["kind"] == "activations" else 0.02, _gen(seed, "w"))}
    if case["kind"] in ("smoothed", "activations"):
        s["peak"] = _uniform((case["k"],), 0.5, 4.0, _gen(seed, "peak"))
    return s


# ---- one pass -------------------------------------------------------------------------------------------------------
def _run_verify(s):
    case, model, kv, buf = s["case"], s["model"], s["kv"], s["buf"]
    if case["commit"]:
        kv.seq_len.copy_(s["lens"])     # the scheduler's lengths of the sequences in this step
    out = {"k": kv.k, "v": kv.v, "seq_len": kv.seq_len, "status": buf.status, "logits": buf.logits}
    if case["entry"] == "host":
        h = s["host"]
        s["plan"].run_host(h["tokens"], h["accept_len"], h["bonus"], block_len_host=h["block_len"],
                           parents_host=h["parents"], accept_path_host=h["path"], status_host=h["status"])
        out.update({n: h[n] for n in ("accept_len", "bonus", "path")})
    else:
        if s["plan"] is not None:
            s["plan"].launch()
        else:
            Q.quasar_verify(model, kv, buf)
        out.update({"accept_len": buf.accept_len, "bonus": buf.bonus, "path": buf.accept_path})
    if case["commit"]:
        if "whole" in s:
            buf.accept_len.copy_(s["whole"])
        Q.quasar_kv_commit(model, kv, buf, tree=case["tree"])
    return out


def run(s):
    case = s["case"]
    op = case["op"]
    if op == "verify":
        return _run_verify(s)
    if op == "linear":
        if case["static"]:
            return Q.quasar_linear_static(s["x"], s["w"], s["delta"], s["out"], residual=s["res"])
        return Q.quasar_linear(s["x"], s["w"], s["delta"], residual=s["res"], out_f32=case["f32"],
                               workspace=s["workspace"], out=s["out"])
    if op == "w8a8":
        return Q.quasar_linear_w8a8(s["x"], s["smooth"], s["w"], s["delta"], residual=s["res"], out_f32=case["f32"])
    if op == "w4":
        return Q.quasar_linear_w4(s["x"], s["w"], s["delta"], residual=s["res"], out_f32=case["f32"])
    if op == "quantize":
        if case["kind"] == "int8":
            return Q.quasar_quantize(s["w"])
        if case["kind"] == "int4":
            return Q.quasar_quantize_int4(s["w"])
        if case["kind"] == "activations":
            return Q.quasar_quantize_activations(s["w"], s["peak"])
        factors = Q.quasar_smoothing_factors(s["peak"], s["w"])
        return (factors,) + Q.quasar_quantize_weights_smoothed(s["w"], factors)
    draft = Q.quasar_ngram_draft(s["history"], s["hist_len"], case["rows"] - 1, 1, 3)
    taken = Q.quasar_accept_stochastic(s["logits"], s["tokens"], s["block_len"], s["q"], 0.8, s["r_accept"], s["r_sample"])
    return {"draft": draft, "taken": taken}


# ---- what a pass cannot do without ----------------------------------------------------------------------------------
def work(case):
    op = case["op"]
    if op == "verify":
        shape = synth.SHAPES[case["model"]]
        lens, blocks = _prefixes(case), _block_lens(case)
        rows, elem = sum(blocks), 2 if case["weights"] == "bf16" else 1
        weights = shape.weight_elems()
        kv_row = 2 * shape.n_layers * shape.kv_dim * 2
        bytes_ = weights * elem + (sum(lens) + rows) * kv_row + rows * shape.hidden * 2
        if elem == 1:
            bytes_ += 4 * (shape.n_layers * sum(n for name, n, _ in shape.linear_shapes() if name != "lm_head") + shape.vocab)
        if case["logits"]:
            bytes_ += rows * shape.vocab * 4
        pairs = sum(t * p + t * (t + 1) // 2 for p, t in zip(lens, blocks))
        return {"bytes": bytes_, "flops": 2 * rows * weights + 4 * pairs * shape.q_dim * shape.n_layers}
    if op == "sample":
        rows = case["batch"] * case["rows"]
        return {"bytes": rows * case["vocab"] * 4 * (2 if case["with_q"] else 1) + case["batch"] * case["history"] * 3,
                "flops": 4 * rows * case["vocab"]}
    n, k = case["n"], case["k"]
    if op == "quantize":
        out = n * k // 2 + n * k // 32 if case["kind"] == "int4" else n * k + 4 * n
        return {"bytes": 2 * n * k + out, "flops": 3 * n * k}
    m = case["m"]
    weights = n * k // 2 + n * k // 32 if op == "w4" else n * k + 4 * n
    if op == "linear" and case["weights"] == "bf16":
        weights = 2 * n * k
    bytes_ = weights + 2 * m * k + m * n * (4 if case["f32"] else 2) + (2 * m * n if case["residual"] else 0)
    return {"bytes": bytes_, "flops": 2 * m * n * k}


def tolerance(case):
    if case["op"] == "quantize":
        return "exact"      # codes and step sizes are defined bit for bit
    if case["op"] == "sample":
        return "exact"      # whole numbers
    if case["op"] == "verify":
        # bf16 between the steps of the pass.  Two sums of one residual row in different orders round apart by about 2^-9 of
        # the row (rms 1.1e-3), twice a layer on both sides: sqrt(4 * 36) * 1.1e-3 = 1.4e-2 on the stream of 36 layers, and
        # the other bf16 tensors add to it (2.0e-2 between the two forms of the 8B pass).  int8 activations turn such a
        # rounding into a quantisation step now and then.
        small = case["model"].startswith("tiny")
        return {"rel": 3e-2 if not small else 2e-2 if case["weights"] == "w8a8" else 1e-2}
    if case["f32"]:
        return {"rel": 5e-5}    # fp32 sums of up to 17,408 products, on tensor cores that truncate each partial sum
    return {"rel": 4e-3}        # one rounding to bf16

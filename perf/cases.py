"""Timed cases of the retrieval path: what a program that uses this package has it do, over the real range of sizes.

A case names one path through the public binding and its sizes:
  question    rekv_question: retrieve, gather and attend for a batch of questions, all layers at once
  layers      rekv_question_layer for one layer after the other, as a decoder that makes its queries layer by layer calls it
  decode      rekv_attend_full_layer for one layer after the other: one generated token over the gathered context
  full        rekv_gather + rekv_attend_full: Eq. 3 with the question's own K/V, all layers; top_k = 0 makes it an
              encoding step (Eq. 1: the incoming frame's tokens over the window and themselves)
  ingest      a stream from its first frame on: rekv_create, rekv_append_frame for every frame, one question, rekv_destroy
  external    rekv_retrieve_external: scores and selection on the embeddings of a CLIP-like encoder

Inputs are the seeded K/V and Q of the package's generator (a per-frame offset makes the frames separable).
"""
import torch

from paper_2503_00540_b200 import rekv, synth

D = 128
PAGE_LIMIT = 20.3e9   # bytes of K/V pages of the largest cache: one hour at 0.5 fps, 28 layers, 4 KV heads, 196 tokens
HOST_LIMIT = 4.5e9    # bytes of pinned host memory of the largest offloaded cache here

BASE = dict(L=28, Hq=28, Hkv=4, Nf=196, T=1800, W=8, k=64, b=1, nQ=1, q_lo=32, q_hi=32, history=0, rope="none", tail=0,
            fp8=False, E=0)


def case(path, **kw):
    return dict(BASE, path=path, **kw)


def listed():
    return [
        # the smallest question: one layer, frames of 16 tokens; launches and latency are everything
        dict(case("question", L=1, Hq=8, Hkv=2, Nf=16, T=64, W=4, k=8, q_lo=16, q_hi=16), name="question_tiny"),
        # the ordinary question: one-hour stream, a sentence of 32 tokens
        dict(case("question"), name="question_1800f"),
        # a short question (one row tile per KV head) with block retrieval over an odd number of frames
        dict(case("question", T=1201, b=8, q_lo=10, q_hi=10), name="question_short_block8"),
        # a server's batch: 16 independent questions of 24 to 64 tokens on one stream
        dict(case("question", k=32, nQ=16, q_lo=24, q_hi=64), name="question_batch16"),
        # a decoder's way: one layer at a time
        dict(case("layers"), name="layers_1800f"),
        # the tokens after the question: one token through all layers, rotary embedding at consecutive positions
        dict(case("decode", T=600, q_lo=1, q_hi=1, history=47, rope="consecutive"), name="decode_rope"),
        # the question's prefill with its own K/V and rotary embedding
        dict(case("full", T=600, rope="consecutive"), name="full_rope"),
        # encoding one incoming frame over the local window
        dict(case("full", T=64, k=0, q_lo=196, q_hi=196, rope="consecutive"), name="encode_frame"),
        # a ten-minute stream ingested and asked about
        dict(case("ingest", T=300), name="ingest_300f"),
        # K/V in pinned host memory, the last frames in HBM
        dict(case("question", T=320, tail=64), name="offload_320f"),
        # the large model's heads and layers, host tier held in FP8
        dict(case("question", L=80, Hq=64, Hkv=8, T=128, k=32, q_lo=64, q_hi=64, tail=32, fp8=True), name="offload_large_fp8"),
        # the external retriever on SigLIP-sized embeddings
        dict(case("external", L=28, Nf=1, T=1800, nQ=4, E=1152), name="external_1800f"),
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    """A case of the same ranges: 4 to 40 layers, the three head groupings, 16 to 256 tokens per frame, streams of
    64 to 1800 frames, questions of 1 to 64 tokens, up to 64 retrieved frames."""
    while True:
        path = rng.choice(("question", "question", "question", "layers", "decode", "full", "encode", "ingest", "offload", "external"))
        Hq, Hkv = rng.choice(((8, 2), (28, 4), (64, 8)))
        c = case(path, L=_log(rng, 4, 40), Hq=Hq, Hkv=Hkv, Nf=_log(rng, 16, 256), T=_log(rng, 64, 1800), W=rng.randint(1, 12),
                 k=_log(rng, 8, 64))
        c["q_lo"] = c["q_hi"] = _log(rng, 1, 64)
        if path == "question":
            if rng.random() < 0.4:
                c.update(nQ=_log(rng, 2, 16), q_lo=rng.randint(1, 32), k=min(c["k"], 32))
                c["q_hi"] = c["q_lo"] + rng.randint(0, 32)
            elif rng.random() < 0.3:
                c["b"] = rng.choice((2, 4, 8))
                c["k"] = -(-c["k"] // c["b"]) * c["b"]
        elif path == "decode":
            c.update(q_lo=1, q_hi=1, history=_log(rng, 8, 150), rope=rng.choice(("none", "consecutive", "static")))
        elif path == "full":
            c.update(rope=rng.choice(("none", "consecutive", "static")))
        elif path == "encode":
            c.update(path="full", k=0, q_lo=c["Nf"], q_hi=c["Nf"], T=min(c["T"], 128), rope=rng.choice(("none", "consecutive")))
        elif path == "ingest":
            c["T"] = min(c["T"], 400)
        elif path == "offload":
            c.update(path="question", T=min(c["T"], 400), tail=32, fp8=rng.random() < 0.5)
        elif path == "external":
            c.update(Hq=28, Hkv=4, Nf=1, nQ=rng.randint(1, 16), E=4 * rng.randint(64, 512))
        pages = c["T"] * c["L"] * _page(c)
        if pages > (HOST_LIMIT if c["tail"] else PAGE_LIMIT / 4 if path == "ingest" else PAGE_LIMIT):
            continue
        if c["nQ"] * c["k"] > 16 * 32 and path != "external":
            continue
        return c


def _page(c):
    return c["Hkv"] * 2 * c["Nf"] * D * 2


def _lengths(c):
    return synth.question_lengths(2503, c["nQ"], c["q_lo"], c["q_hi"])


def _cu(lengths):
    cu = [0]
    for n in lengths:
        cu.append(cu[-1] + n)
    return cu


def _context(c, lengths):
    n_q = sum(lengths)
    flags = (rekv.FLAG_HOST_FP8 if c["fp8"] else 0) | (rekv.FLAG_ROPE_STATIC if c["rope"] == "static" else 0)
    return rekv.ReKV(c["L"], c["Hq"], c["Hkv"], D, c["Nf"], c["T"], c["W"], hbm_tail_frames=c["tail"], max_q_tokens=n_q,
                     max_topk=c["k"], max_questions=c["nQ"], flags=flags, block_frames=c["b"],
                     max_self_tokens=n_q + c["history"] * c["nQ"] if c["path"] in ("decode", "full") else 0,
                     rope_theta=0.0 if c["rope"] == "none" else 1e6, ext_embed_dim=c["E"])


def _frame(c, seed, which, f):
    return synth.frame(seed, which, f, c["L"], c["Nf"], c["Hkv"], D, 0.5, "cuda:0")


def _queries(c, seed, first, lengths):
    q = torch.empty((c["L"], sum(lengths), c["Hq"], D), dtype=torch.bfloat16, device="cuda:0")
    at = 0
    for i, n in enumerate(lengths):
        q[:, at:at + n] = synth.question(seed, first + i, c["L"], n, c["Hq"], D, "cuda:0")
        at += n
    return q


def prepare(case, seed):
    c = case
    lengths = _lengths(c)
    s = {"case": c, "cu": _cu(lengths)}
    if c["path"] == "external":
        g = torch.Generator(device="cuda:0").manual_seed(seed)
        s["ctx"] = ctx = _context(c, lengths)
        emb = torch.randn((c["T"], c["E"]), generator=g, device="cuda:0")
        s["q_emb"] = torch.randn((c["nQ"], c["E"]), generator=g, device="cuda:0")
        kv = torch.zeros((c["L"], 1, c["Hkv"], D), dtype=torch.bfloat16, device="cuda:0")
        for f in range(c["T"]):
            ctx.append_frame(kv, kv)
            ctx.set_frame_embedding(f, emb[f])
        return s
    s["q"] = _queries(c, seed, 0, lengths)
    if c["path"] == "ingest":
        s["k"] = [_frame(c, seed, synth.K, f) for f in range(c["T"])]
        s["v"] = [_frame(c, seed, synth.V, f) for f in range(c["T"])]
        return s
    s["ctx"] = ctx = _context(c, lengths)
    for f in range(c["T"]):
        ctx.append_frame(_frame(c, seed, synth.K, f), _frame(c, seed, synth.V, f))
    if c["path"] == "layers":
        s["out"] = torch.empty_like(s["q"])
    if c["path"] in ("decode", "full"):
        own = [n + c["history"] for n in lengths]
        s["cu_self"] = _cu(own)
        # the questions' own keys and values: one "frame" of that many tokens
        s["k"], s["v"] = (synth.frame(seed, w, c["T"], c["L"], sum(own), c["Hkv"], D, 0.5, "cuda:0") for w in (synth.K, synth.V))
        s["idx"] = ctx.retrieve(s["q"], s["cu"], c["k"], c["T"])[0]
    if c["path"] == "decode":
        s["out"] = torch.empty_like(s["q"])
        ctx.gather(s["idx"], c["nQ"], c["k"], c["T"])
    return s


def run(state):
    s, c = state, state["case"]
    path, cu = c["path"], s["cu"]
    if path == "question":
        return s["ctx"].question(s["q"], cu, c["k"], c["T"])
    if path == "layers":
        ctx, q, out = s["ctx"], s["q"], s["out"]
        for l in range(c["L"]):
            ctx.question_layer(l, q[l], cu, c["k"], c["T"], out=out[l])
        return out
    if path == "decode":
        ctx, q, k, v, out = s["ctx"], s["q"], s["k"], s["v"], s["out"]
        for l in range(c["L"]):
            ctx.attend_full_layer(l, q[l], k[l], v[l], cu, s["cu_self"], out=out[l])
        return out
    if path == "full":
        s["ctx"].gather(s["idx"], c["nQ"], c["k"], c["T"])
        return s["ctx"].attend_full(s["q"], s["k"], s["v"], cu, s["cu_self"])
    if path == "ingest":
        ctx = _context(c, _lengths(c))
        for k, v in zip(s["k"], s["v"]):
            ctx.append_frame(k, v)
        idx, _, scores = ctx.retrieve(s["q"], cu, c["k"], c["T"], want_scores=True)
        ctx.gather(idx, c["nQ"], c["k"], c["T"])
        out = ctx.attend(s["q"], cu)
        ctx.close()
        return out, idx, scores
    idx, _, scores = s["ctx"].retrieve_external(s["q_emb"], c["k"], c["T"], 0.07, want_scores=True)
    return idx, scores


def work(case):
    c = case
    L, nQ, n_q = c["L"], c["nQ"], sum(_lengths(c))
    if c["path"] == "external":
        return {"bytes": 4.0 * (c["T"] * c["E"] + nQ * (c["E"] + c["T"]) + L * nQ * c["k"]), "flops": 2.0 * c["T"] * c["E"] * (nQ + 1)}
    n_cand = max(c["T"] - c["W"], 0) // c["b"] * c["b"]
    k_eff = min(c["k"], n_cand)
    ctx_frames = k_eff + c["T"] - n_cand
    # each context frame's page once (the trailing frames are shared by the batch), queries in and outputs out
    b = L * (nQ * k_eff + c["T"] - n_cand) * _page(c) + 2.0 * L * n_q * c["Hq"] * D * 2
    f = 4.0 * L * n_q * c["Hq"] * ctx_frames * c["Nf"] * D
    if c["path"] in ("question", "layers", "ingest"):
        b += 4.0 * L * c["T"] * c["Hkv"] * D   # the representatives
        f += 2.0 * L * c["T"] * c["Hkv"] * D * nQ
    if c["path"] in ("decode", "full"):
        b += L * sum(n + c["history"] for n in _lengths(c)) * c["Hkv"] * D * 2 * 2
        f += sum(4.0 * L * c["Hq"] * D * n * (c["history"] + (n + 1) / 2) for n in _lengths(c))
    if c["path"] == "ingest":
        b += 2.0 * L * c["T"] * _page(c) + 4.0 * L * c["T"]
        f += L * c["T"] * _page(c) / 4.0
    return {"bytes": float(b), "flops": float(f)}


def tolerance(case):
    # scores: fp32 sums; a selection may differ where two scores tie to rounding
    if case["path"] == "external":
        return {"rel": 1e-5, "differ": 0.01}
    # bf16 operands and results, P in bf16: 1.9e-3 normwise and 6.2e-3 of the rms at most against fp64 sums over
    # the same context (two layers of each listed case)
    return {"rel": 7e-3, "max": 0.025, "differ": 0.01}

"""Performance cases of the library: what its users have it do, through the public Python entry points.

A case is a dict of plain values.  ``kind`` says which calls one pass makes:

  roundtrip   encode a batch's KV cache and decode it again (spill and restore of a prefill)
  decode      decode a cache that was encoded before (restore alone)
  adaptive    roundtrip with the surprisal-adaptive step (both calls also take the tokens)
  rotq        roundtrip with the rotated fixed-rate quantiser
  dense       roundtrip with the full-vocabulary predictor
  linear      roundtrip with the linear-embedding predictor
  append      n decode-time steps of S sessions, then the flush at the end of the generation
  topk        top-K softmax of S*n rows with every output
  dedup       log2 P of the sessions' tokens, their common prefixes, their clusters

The encoders place chunks in the order in which they are finished, so offsets and the order of the
payload are not part of a pass's result; the chunks' sizes are, and their contents are read back by
the decode of the same pass.
"""
import math

import torch

import paper_2604_15356_b200 as plc


def listed():
    return [
        # The tiny configuration: one short session on a two-stream model; latency and launches count.
        _case("roundtrip-tiny", "roundtrip", S=1, n=512, L=1, H=1, d=64, V=256, K=16, pp=12.0, alpha=0.0),
        # One short prompt of odd length, partly shared with an earlier session (position ranges), odd vocabulary.
        _case("roundtrip-short-ragged", "roundtrip", S=3, n=333, L=4, H=8, d=64, V=50001, K=50, chunk=64, ranges=True),
        # The headline shape (32 heads of 128, Zipf-skewed candidates), half of its layers: a serving node's prefill batch.
        _case("roundtrip-prefill", "roundtrip", S=4, n=4096, L=16, H=32, d=128, V=32000, K=64, f16=True),
        # Restore of one very long context: four layers of the long-context shape.
        _case("decode-longctx", "decode", S=1, n=131072, L=4, H=8, d=128, V=32000, K=64, pp=20.0, alpha=0.0),
        # Variable-precision cache of a mid-sized batch.
        _case("roundtrip-adaptive", "adaptive", S=2, n=2048, L=8, H=8, d=128, V=32000, K=64),
        # Fixed-rate records (4 bits) of a mid-sized batch.
        _case("roundtrip-rotq", "rotq", S=4, n=1000, L=8, H=8, d=128, V=32000, K=64, bits=4),
        # Full-vocabulary prediction of a prefill, tensor-core bound.
        _case("roundtrip-dense", "dense", S=1, n=8192, L=4, H=8, d=128, V=32000, pp=20.0, alpha=0.0),
        # Linear-embedding prediction of a short batch.
        _case("roundtrip-linear", "linear", S=4, n=512, L=8, H=8, d=128, V=32000, dm=4096),
        # Generation with a full batch: the append configuration over one chunk and a quarter.
        _case("append-batch", "append", S=256, n=40, L=32, H=8, d=128, V=32000, K=64, chunk=32, pp=12.0, alpha=0.0),
        # Generation of a single session with a large vocabulary: latency of one token's step.
        _case("append-single", "append", S=1, n=40, L=16, H=8, d=128, V=128256, K=64, chunk=32, pp=12.0, alpha=0.0),
        # Candidate selection by itself on the large vocabulary.
        _case("topk-large-vocab", "topk", S=1, n=4096, V=128256, K=64),
        # Prefix deduplication of a batch of sessions.
        _case("dedup-sessions", "dedup", S=64, n=384, V=128256, pp=12.0, alpha=0.0),
    ]


def _case(name, kind, **over):
    c = {"kind": kind, "S": 1, "n": 1, "L": 1, "H": 1, "d": 128, "V": 32000, "K": 64, "pp": 15.0, "alpha": 1.1, "delta": 0.02,
         "chunk": 256, "f16": False, "ranges": False, "bits": 0, "dm": 0}
    c.update(over)
    return dict(c, name=name) if name else c


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case: the kinds above over the sizes, types and options that the listed ones stand for."""
    kind = rng.choice(["roundtrip", "roundtrip", "roundtrip", "decode", "adaptive", "rotq", "dense", "linear", "append", "append",
                       "topk", "dedup"])
    V = _log_int(rng, 256, 131072)
    if rng.random() < 0.6:
        V = (V + 7) // 8 * 8                              # vocabularies are usually padded; some are not
    c = _case("", kind, V=V, pp=rng.choice([6.0, 12.0, 15.0, 20.0, 40.0]), alpha=rng.choice([0.0, 1.1]),
              delta=rng.choice([0.005, 0.02, 0.02, 0.08]), f16=rng.random() < 0.5,
              K=min(V, rng.choice([16, 32, 50, 64, 64, 64, 100, 128])))
    c["pp"] = min(c["pp"], V / 4.0)
    if kind in ("topk", "dedup"):
        rows = _log_int(rng, 1, min(32768, (1 << 31) // V))
        c["S"] = min(rows, _log_int(rng, 1, 128))
        c["n"] = max(1, rows // c["S"])
        return c
    c["d"] = rng.choice([32, 64, 128, 128, 128, 128, 256])
    c["H"] = rng.choice([1, 2, 4, 8, 8, 8, 16, 32])
    c["L"] = _log_int(rng, 1, 32)
    while 2 * c["L"] * c["H"] * V * c["d"] > (1 << 32) and c["L"] > 1:      # candidate tables of at most 8 GB
        c["L"] = (c["L"] + 1) // 2
    while 2 * c["L"] * c["H"] * V * c["d"] > (1 << 32):
        c["H"] = (c["H"] + 1) // 2
    W = 2 * c["L"] * c["H"]
    if kind == "append":
        c["chunk"] = 32
        c["n"] = rng.randint(8, 48)
        c["S"] = _log_int(rng, 1, max(1, min(256, (1 << 24) // (W * c["d"]))))
        return c
    c["chunk"] = rng.choice([64, 128, 256, 256])
    if kind == "rotq":
        c["bits"] = rng.choice([2, 3, 4, 6])
    if kind in ("dense", "linear"):
        c["H"] = min(c["H"], 16)
        c["L"] = min(c["L"], 4)
        c["dm"] = 64 * rng.randint(8, 64) if kind == "linear" else 0
        most = min(8192, int(4e12 / (2.0 * max(V, 2048) * 2 * c["H"] * c["d"] * c["L"])))
    else:
        # at most about 1e11 multiply-adds of the mixture, 4 GB of logits, 2 GB of KV
        most = min(65536, int(1e11 / (W * c["d"] * c["K"])), (1 << 31) // V, (1 << 30) // (W * c["d"]))
    rows = _log_int(rng, 16, max(17, most))
    c["S"] = min(rows, _log_int(rng, 1, 16))
    c["n"] = max(1, rows // c["S"])
    c["ranges"] = kind == "roundtrip" and c["n"] > 8 and rng.random() < 0.4
    return c


# ---- inputs -------------------------------------------------------------------------------------

def _rows_at_once(V):
    return max(1, (1 << 28) // V)


def _logits(c, rows, gen):
    """float16 [rows][V] next-token logits of about the stated perplexity and tokens [rows] drawn from them:
    tau * (-alpha ln(1 + rank) + N(0,1)), the rank being one permutation of the vocabulary for all rows
    (frequent tokens are likely everywhere), tau found by bisection on a few rows."""
    V, dev = c["V"], "cuda"
    prior = 0.0
    if c["alpha"]:
        prior = -c["alpha"] * torch.log1p(torch.randperm(V, generator=gen, device=dev).float())
    probe = torch.randn(16, V, generator=gen, device=dev) + prior
    lo, hi = 0.0, 64.0
    for _ in range(20):
        mid = 0.5 * (lo + hi)
        lp = torch.log_softmax(probe * mid, 1)
        if float(-(lp.exp() * lp).sum(1).mean()) > math.log(c["pp"]):
            lo = mid
        else:
            hi = mid
    tau = 0.5 * (lo + hi)
    out = torch.empty(rows, V, dtype=torch.float16, device=dev)
    tokens = torch.empty(rows, dtype=torch.int32, device=dev)
    step = _rows_at_once(V)
    for r in range(0, rows, step):
        x = torch.randn(min(step, rows - r), V, generator=gen, device=dev)
        out[r:r + step] = (x + prior).mul_(tau)
        x = torch.softmax(out[r:r + step].float(), 1)
        q = torch.empty_like(x).exponential_(generator=gen)
        tokens[r:r + step] = x.div_(q).argmax(1).to(torch.int32)
    return out, tokens


def _tables(c, gen):
    T = torch.empty(c["L"], 2, c["H"], c["V"], c["d"], dtype=torch.float16, device="cuda")
    for l in range(c["L"]):
        T[l].normal_(generator=gen)
    return T


def _kv(c, T, tokens, gen):
    """[L][2][S][H][n][d] float16: the token's own row plus a little noise."""
    S, n, H, d = c["S"], c["n"], c["H"], c["d"]
    kv = torch.empty(c["L"], 2, S, H, n, d, dtype=torch.float16, device="cuda")
    at = tokens.to(torch.int64)
    for l in range(c["L"]):
        for a in range(2):
            rows = T[l, a].index_select(1, at)                                   # [H][S*n][d]
            rows += torch.empty_like(rows).normal_(0.0, 0.05, generator=gen)
            kv[l, a].copy_(rows.view(H, S, n, d).transpose(0, 1))
    return kv


def _kv_linear(c, E, A, bias, tokens, gen):
    S, n, H, d = c["S"], c["n"], c["H"], c["d"]
    kv = torch.empty(c["L"], 2, S, H, n, d, dtype=torch.float16, device="cuda")
    emb = E[tokens.to(torch.int64)]
    for l in range(c["L"]):
        for a in range(2):
            rows = (emb @ A[l, a].reshape(H * d, -1).t()).view(S * n, H, d) + bias[l, a]
            rows += torch.empty_like(rows).normal_(0.0, 0.05, generator=gen)
            kv[l, a].copy_(rows.view(S, n, H, d).transpose(1, 2))
    return kv


def _share_prefixes(c, logits, tokens, host):
    """Sessions 1.. continue a random prefix of an earlier session (same tokens, same distributions there)."""
    S, n = c["S"], c["n"]
    logits, tokens = logits.view(S, n, c["V"]), tokens.view(S, n)
    for s in range(1, S):
        p = int(torch.randint(0, s, (1,), generator=host))
        m = int(torch.randint(0, n + 1, (1,), generator=host)) * 3 // 4
        if m:
            logits[s, :m] = logits[p, :m]
            tokens[s, :m] = tokens[p, :m]


def prepare(case, seed):
    c = case
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    host = torch.Generator().manual_seed(int(seed))
    S, n, L, H, d, V, K = (c[k] for k in ("S", "n", "L", "H", "d", "V", "K"))
    s = {"case": c}
    logits, tokens = _logits(c, S * n, gen)
    s["logits"], s["tokens"] = logits.view(S, n, V), tokens.view(S, n)
    if c["kind"] in ("topk", "dedup"):
        if c["kind"] == "dedup":
            _share_prefixes(c, logits, tokens, host)
            s["lens"] = torch.randint(max(1, n // 2), n + 1, (S,), generator=host).to(torch.int32).cuda()
        torch.cuda.empty_cache()
        s["ctx"] = plc.Context(torch.zeros(1, 2, 1, V, 32, dtype=torch.float16, device="cuda"), K, c["delta"])
        return s
    out_dtype = plc.OUT_F16 if c["f16"] else plc.OUT_F32
    if c["kind"] == "linear":
        dm = c["dm"]
        E = torch.empty(V, dm, dtype=torch.float16, device="cuda").normal_(generator=gen)
        A = torch.empty(L, 2, H, d, dm, dtype=torch.float16, device="cuda").normal_(0.0, dm ** -0.5, generator=gen)
        bias = torch.empty(L, 2, H, d, dtype=torch.float16, device="cuda").normal_(0.0, 0.1, generator=gen)
        kv = _kv_linear(c, E, A, bias, tokens, gen)
        torch.cuda.empty_cache()
        ctx = plc.Context.linear(E, A, bias, c["delta"], chunk_pos=c["chunk"], out_dtype=out_dtype)
    else:
        T = _tables(c, gen)
        kv = _kv(c, T, tokens, gen)
        torch.cuda.empty_cache()
        variant = plc.PRED_DENSE if c["kind"] == "dense" else plc.PRED_TOPK
        adaptive = (6, 4, math.log2(c["pp"])) if c["kind"] == "adaptive" else None
        ctx = plc.Context(T, K, c["delta"], chunk_pos=c["chunk"], variant=variant, out_dtype=out_dtype, adaptive=adaptive)
    s["ctx"] = ctx
    if c["kind"] == "append":
        s["kv_steps"] = [kv[:, :, :, :, i].contiguous() for i in range(n)]       # [L][2][S][H][d] a step
        s["logit_steps"] = [s["logits"][:, i].contiguous() for i in range(n)]
        del s["logits"], kv
        s["batch"] = ctx.new_session_batch(S, ctx.max_chunks(n), 2 * S * n * ctx.W * d + S * ctx.W * ctx.max_chunks(n) * 160)
        return s
    s["kv"] = kv
    s["out"] = torch.zeros(kv.shape, dtype=torch.float16 if c["f16"] else torch.float32, device="cuda")
    ctx.reserve(S * n)
    if c["kind"] == "rotq":
        s["params"] = ctx.rotq_params(c["bits"], torch.randint(0, 2, (d,), generator=host).tolist())
        s["records"] = torch.zeros(S * ctx.W * n * ctx.rotq_record_bytes(c["bits"]), dtype=torch.uint8, device="cuda")
        return s
    mc = ctx.max_chunks(n)
    s["streams"] = plc.StreamSet(S * ctx.W, mc, 2 * S * n * ctx.W * d + S * ctx.W * mc * 160)
    s["begin"] = s["end"] = None
    if c["ranges"]:
        b = torch.randint(0, n // 2, (S,), generator=host)
        e = torch.randint(n // 2, n + 1, (S,), generator=host)
        e[0], b[-1] = n, 0
        s["begin"], s["end"] = b.to(torch.int32).cuda(), e.to(torch.int32).cuda()
    if c["kind"] == "decode":
        ctx.encode(kv, s["logits"], s["streams"])
        del s["kv"]
    return s


# ---- one pass -----------------------------------------------------------------------------------

def run(state):
    s = state
    c, ctx = s["case"], s["ctx"]
    kind = c["kind"]
    if kind == "topk":
        return ctx.topk_softmax(s["logits"], s["tokens"])
    if kind == "dedup":
        logp2 = ctx.topk_softmax(s["logits"], s["tokens"], want=("logp2",))["logp2"].view(c["S"], c["n"])
        lcp, dT, parent, shared = ctx.prefix_dedup(s["tokens"], s["lens"], logp2)
        return [logp2, lcp, dT, parent, shared, *ctx.prefix_clusters(lcp, dT, 16.0)]
    if kind == "append":
        batch = s["batch"]
        batch.c.steps = 0                                  # a new generation in the same buffers
        batch.streams.total_bytes.zero_()
        for kv, logits in zip(s["kv_steps"], s["logit_steps"]):
            ctx.append_step(batch, kv, logits)
        ctx.append_flush(batch)
        return {"open_sym": batch.open_sym, "open_q": batch.open_q, "chunk_bytes": batch.streams.chunk_bytes,
                "total_bytes": batch.streams.total_bytes}
    if kind == "rotq":
        ctx.encode_rotq(s["kv"], s["logits"], s["params"], s["records"])
        ctx.decode_rotq(s["records"], s["logits"], s["params"], s["out"])
        return {"records": s["records"], "kv": s["out"]}
    st, tokens = s["streams"], s["tokens"] if kind == "adaptive" else None
    if kind != "decode":
        st.total_bytes.zero_()
        ctx.encode(s["kv"], s["logits"], st, s["begin"], s["end"], tokens=tokens)
    ctx.decode(st, s["logits"], s["out"], s["begin"], s["end"], tokens=tokens)
    return {"chunk_bytes": st.chunk_bytes, "total_bytes": st.total_bytes, "kv": s["out"]}


# ---- what a pass cannot do without, and how far results may differ ------------------------------

def work(case):
    """Every call of a pass reads its inputs once (of the candidate tables at most the rows that the
    positions name) and writes its outputs once; the arithmetic is the predictor's."""
    c = case
    rows, V = c["S"] * c["n"], c["V"]
    logits = 2.0 * rows * V
    if c["kind"] == "topk":
        return {"bytes": logits + rows * (8.0 * c["K"] + 16), "flops": 2.0 * rows * V}
    if c["kind"] == "dedup":
        return {"bytes": logits + rows * 12.0 + c["S"] ** 2 * 8.0, "flops": 2.0 * rows * V}
    W, d = 2 * c["L"] * c["H"], c["d"]
    coded = rows * 0.5 if c["ranges"] else float(rows)     # ranges cover between a half and all of a session, on average
    if c["ranges"]:
        logits *= 0.5
    comps = coded * W * d
    rate = c["bits"] / 8.0 if c["kind"] == "rotq" else math.log2(4.0 / c["delta"]) / 8.0   # bytes a component
    out = 2.0 if c["f16"] else 4.0
    calls = 1 if c["kind"] in ("decode", "append") else 2
    if c["kind"] == "dense":
        model, flops = 2.0 * W * V * d, 2.0 * rows * V * W * (d + 1)
    elif c["kind"] == "linear":
        model = 2.0 * c["dm"] * (V + W * d) + 2.0 * W * V
        flops = 2.0 * rows * (V * c["dm"] + V * W + c["dm"] * W * d)
    else:
        model, flops = min(2.0 * W * V * d, 2.0 * comps * c["K"]), 2.0 * comps * c["K"]
        if c["kind"] == "append":
            model = c["n"] * min(2.0 * W * V * d, 2.0 * c["S"] * W * d * c["K"])
    if c["kind"] == "append":                              # symbols go to the open chunk and come back once
        return {"bytes": logits + model + comps * (2.0 + 8.0 + rate), "flops": flops}
    if c["kind"] == "decode":
        return {"bytes": logits + model + comps * (rate + out), "flops": flops}
    return {"bytes": calls * (logits + model + comps * rate) + comps * (2.0 + out), "flops": calls * flops}


def tolerance(case):
    kind = case["kind"]
    if kind in ("topk", "dedup"):
        return {"rel": 1e-5}                               # 32-bit sums; the selected set, prefixes and parents are exact
    if kind == "append":
        return "exact"                                     # whole numbers throughout
    if kind in ("dense", "linear"):
        # bf16 contraction: where the prediction's last bits carry a component across a rounding boundary
        # of the quantiser the symbol moves by one step
        return {"rel": 1e-3, "max": 0.25, "differ": 0.01}
    if kind == "rotq":
        return {"rel": 1e-4, "max": 0.1, "differ": 0.002}  # a code may move by one level at a boundary
    return {"rel": 1e-5, "max": 4e-4}                      # 32-bit prediction; the chunks' sizes are exact

"""The work a user of this library has it do, as timed cases through the public Python entry points.

Every case is one operator of include/hils.h on seeded synthetic tensors (paper_2607_02980_b200.workloads: K, V, Q
of unit variance, landmarks = chunk means plus noise, planted needles or queries that drift slowly from token to
token).  The listed sizes are the repository's benchmark configurations and the shapes around them that serving and
training meet: one short sequence, batches of unequal lengths, prompts whose length is no multiple of a chunk, a slice
of a long prompt, the paper's operator form (local window of 512 tokens plus bias), drafts of several tokens.
"""
import math

import numpy as np
import torch

import paper_2607_02980_b200 as hils
from paper_2607_02980_b200 import workloads as wl

S = 64                        # chunk size of every configuration

# Plain fields of a case.  T is the number of tokens in the caches (prefill: of the sequence), pos0 the position of
# the first query token of a slice, M the new tokens per sequence, W the local window, overlap = 1 for queries that
# share most of their chunks with their neighbours (0: independent queries with planted needles).
_DEFAULTS = {"B": 1, "Hq": 32, "Hkv": 8, "d": 128, "K": 16, "W": 1, "bias": False, "dtype": "bf16",
             "pos0": 0, "L": 0, "M": 1, "ragged": False, "overlap": False}


def _case(kind, T, **kw):
    return dict(_DEFAULTS, kind=kind, T=T, **kw)


def listed():
    return [
        # one interactive user, a short conversation: three small launches, latency and host work are everything
        dict(_case("decode", 6000, K=16), name="decode_one_6k"),
        # a small serving batch of unequal lengths on a paged cache, in the paper's form (window 512, bias)
        dict(_case("decode_paged", 16384, B=8, K=32, W=512, bias=True, ragged=True), name="decode_paged_b8_16k"),
        # batched serving at 64K tokens (benchmark configuration 3)
        dict(_case("decode", 65536, B=64, K=32), name="decode_b64_64k"),
        # a few million-token sequences (benchmark configuration 4): long candidate lists, little else
        dict(_case("decode", 1048576, B=4, K=64), name="decode_b4_1m"),
        # verification of four draft tokens per sequence
        dict(_case("decode_multi", 32768, B=16, K=32, M=4, ragged=True), name="decode_multi_b16_32k"),
        # short prompts of a length that fits no tile, prefilled together
        dict(_case("prefill", 1000, B=3, K=16), name="prefill_b3_1000"),
        # benchmark configuration 1
        dict(_case("prefill", 16384, K=16), name="prefill_16k"),
        # benchmark configuration 2, the largest prefill
        dict(_case("prefill", 131072, K=32), name="prefill_128k"),
        # chunked prefill: a slice of a long prompt at an odd offset, the paper's form, neighbours that share chunks
        dict(_case("prefill_at", 50000, L=2048, pos0=47777, K=32, W=512, bias=True, overlap=True), name="slice_2k_of_50k"),
        # one training step of the operator: forward, then the gradients of every input
        dict(_case("train", 16384, K=16, bias=True), name="train_16k"),
        # chunk summaries of filled caches (the landmarks and biases of all chunks)
        dict(_case("summary", 65536, B=8, ragged=True), name="summary_b8_64k"),
        # fp32 on small shapes: the reference precision, benchmark configuration 0
        dict(_case("prefill", 2048, Hq=1, Hkv=1, d=64, K=4, dtype="f32"), name="prefill_f32_2k"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["decode", "decode", "decode_paged", "decode_multi", "prefill", "prefill", "prefill_at", "train",
                       "summary", "prefill_f32"])
    paper = rng.random() < 0.4                            # the paper's form: window and bias
    W, bias = (rng.choice([128, 512]), True) if paper else (1, rng.random() < 0.25)
    Hq, Hkv = rng.choice([(32, 8), (32, 8), (16, 4), (8, 2)])
    common = dict(Hq=Hq, Hkv=Hkv, W=W, bias=bias)
    if kind in ("decode", "decode_paged", "decode_multi"):
        if rng.random() < 0.25:
            common.update(Hq=64, Hkv=8)                   # eight query heads per KV head
        most = 64 * 65536 if kind == "decode" else 16 * 65536
        T = _log(rng, 1024, 1048576 if kind == "decode" else 131072)
        B = _log(rng, 1, max(1, min(64, most // T)))
        if kind == "decode_paged":
            T = (T + S - 1) // S * S
        return _case(kind, T, B=B, K=rng.choice([16, 32, 64]), M=rng.choice([2, 4]) if kind == "decode_multi" else 1,
                     ragged=rng.random() < 0.6, **common)
    if kind == "prefill":
        T = _log(rng, 200, 100000)
        B = _log(rng, 1, max(1, min(8, 65536 // T)))
        return _case(kind, T, B=B, K=rng.choice([16, 32]), overlap=rng.random() < 0.3, **common)
    if kind == "prefill_at":
        L = _log(rng, 64, 8192)
        T = max(L, _log(rng, 4096, 131072))
        return _case(kind, T, L=L, pos0=rng.randint(0, T - L), K=rng.choice([16, 32]), overlap=rng.random() < 0.5, **common)
    if kind == "train":
        T = _log(rng, 512, 24000)
        B = _log(rng, 1, max(1, min(4, 16384 // T)))
        return _case(kind, T, B=B, K=rng.choice([8, 16, 32]), overlap=rng.random() < 0.3, **common)
    if kind == "summary":
        T = _log(rng, 1024, 262144)
        B = _log(rng, 1, max(1, min(64, 8 * 65536 // T)))
        return _case(kind, T, B=B, ragged=rng.random() < 0.6, **dict(common, W=1, bias=False))
    Hq, Hkv = rng.choice([(1, 1), (2, 1), (4, 2)])
    return _case("prefill", _log(rng, 200, 4096), Hq=Hq, Hkv=Hkv, d=rng.choice([64, 128]), K=rng.choice([4, 8]), dtype="f32")


# ---------------------------------------------------------------------------------------------------- sizes of a case
def _chunks(c):
    return max(1, c["T"] // S)


def _lengths(c):
    """Tokens of every sequence: all T, or spread over T/4 .. T (a property of the case, not of the seed)."""
    if not c["ragged"]:
        return [c["T"]] * c["B"]
    low = max(c["M"], c["T"] // 4)
    return [c["T"] - (b * 7919 + 13) % (c["T"] - low + 1) for b in range(c["B"])]


def _positions(c):
    """Positions of the query tokens of one sequence (prefill kinds)."""
    return np.arange(c["pos0"], c["pos0"] + (c["L"] or c["T"]), dtype=np.int64)


def _left(pos, W):
    return np.maximum(0, (pos - W + 1) // S) * S


def _config(c, seed):
    return wl.HilsConfig("case", "decode" if c["kind"].startswith("decode") else "prefill", c["B"], c["Hq"], c["Hkv"],
                         c["T"], c["d"], S, c["K"], c["dtype"], int(seed), n_needles=2, window=c["W"])


# ------------------------------------------------------------------------------------------------------------- inputs
def _bias(cfg):
    return wl.make_bias(cfg, "cuda")


def _draft_queries(c, cfg, landmarks, lens):
    """[B, M, Hq, d]: the draft tokens of a sequence retrieve nearly the same chunks (one base query plus noise)."""
    base = wl.make_decode_queries(cfg, landmarks, lens).float()
    g = torch.Generator(device="cuda")
    g.manual_seed(cfg.seed * 1000 + 99)
    noise = torch.randn((c["B"], c["M"], c["Hq"], c["d"]), generator=g, device="cuda")
    return (base[:, None] + 0.3 * noise).to(cfg.torch_dtype())


def _pages(c, cfg, t):
    """[P, Hkv, S, d] pages in a shuffled order; page of chunk (b, n) = table[b, n]."""
    C = _chunks(c)
    g = torch.Generator(device="cuda")
    g.manual_seed(cfg.seed * 1000 + 98)
    table = torch.randperm(c["B"] * C, generator=g, device="cuda")
    where = torch.argsort(table)
    def lay(x):
        return x.view(c["B"], c["Hkv"], C, S, c["d"]).transpose(1, 2).reshape(-1, c["Hkv"], S, c["d"])[where].contiguous()
    return lay(t["k"]), lay(t["v"]), table.view(c["B"], C).to(torch.int32)


def _with_landmark_rows(c, t):
    """A sequence shorter than a chunk has no landmark yet; the tensors still hold one row."""
    if t["landmarks"].shape[2] == 0:
        t["landmarks"] = torch.zeros((c["B"], c["Hkv"], 1, c["d"]), dtype=t["k"].dtype, device="cuda")
    return t


def _decode_state(c, cfg):
    lens = torch.tensor(_lengths(c), dtype=torch.int32, device="cuda")
    t = wl.make_decode_inputs(cfg, "cuda", seq_lens=lens)
    C, B, Hq, Hkv, K, d, M = t["landmarks"].shape[2], c["B"], c["Hq"], c["Hkv"], c["K"], c["d"], c["M"]
    t["bias"] = _bias(cfg) if c["bias"] else None
    lead = (B,) if c["kind"] != "decode_multi" else (B, M)
    if c["kind"] == "decode_multi":
        t["q"] = _draft_queries(c, cfg, t["landmarks"], lens)
    if c["kind"] == "decode_paged":
        t["k"], t["v"], t["table"] = _pages(c, cfg, t)
    # the buffers that a decoding loop keeps from step to step
    t["out"] = torch.empty(lead + (Hq, d), dtype=t["q"].dtype, device="cuda")
    t["lse"] = torch.empty(lead + (Hq,), dtype=torch.float32, device="cuda")
    t["sel"] = torch.empty(lead + (Hkv, K), dtype=torch.int32, device="cuda")
    p = hils.make_params(B=B * M, Hq=Hq, Hkv=Hkv, Hl=Hkv, L=0, T_max=c["T"], C=C, d=d, chunk_size=S, top_k=K,
                         window=c["W"], dtype=1)
    t["ws"] = hils.alloc_workspace(p, True, "cuda") if c["kind"] != "decode_multi" else None
    return t


def _prefill_state(c, cfg):
    extra = dict(overlap_block=16, overlap_noise=0.3, overlap_drift=0.0) if c["overlap"] else {}
    t = _with_landmark_rows(c, wl.make_prefill_inputs(cfg, "cuda", **extra))
    t["bias"] = _bias(cfg) if c["bias"] else None
    if c["bias"] and t["bias"].shape[2] == 0:
        t["bias"] = torch.zeros((c["B"], c["Hkv"], 1), device="cuda")
    if c["kind"] == "prefill_at":
        t["q"] = t["q"][:, :, c["pos0"]:c["pos0"] + c["L"]].contiguous()
    if c["kind"] == "train":
        g = torch.Generator(device="cuda")
        g.manual_seed(cfg.seed * 1000 + 97)
        t["dout"] = torch.randn(t["q"].shape, generator=g, device="cuda").to(t["q"].dtype)
        for n in ("q", "k", "v", "landmarks", "bias"):
            if t[n] is not None:
                t[n].requires_grad_(True)
    elif c["kind"] == "prefill":                          # a prefilling server keeps its workspace
        p = hils.make_params(B=c["B"], Hq=c["Hq"], Hkv=c["Hkv"], Hl=c["Hkv"], L=c["T"], T_max=c["T"],
                             C=t["landmarks"].shape[2], d=c["d"], chunk_size=S, top_k=c["K"], window=c["W"],
                             dtype=0 if c["dtype"] == "f32" else 1)
        t["ws"] = hils.alloc_workspace(p, False, "cuda")
    return t


def _summary_state(c, cfg):
    g = torch.Generator(device="cuda")
    g.manual_seed(cfg.seed * 1000 + 96)
    C = _chunks(c)
    k = torch.randn((c["B"], c["Hkv"], c["T"], c["d"]), generator=g, device="cuda", dtype=torch.bfloat16)
    lq = torch.randn((c["B"], c["Hkv"], C, c["d"]), generator=g, device="cuda", dtype=torch.bfloat16)
    return {"k": k, "lq": lq, "lens": torch.tensor(_lengths(c), dtype=torch.int32, device="cuda"),
            "landmarks": torch.zeros_like(lq), "bias": torch.zeros((c["B"], c["Hkv"], C), device="cuda")}


def prepare(case, seed):
    c = dict(_DEFAULTS, **case)
    cfg = _config(c, seed)
    if c["kind"].startswith("decode"):
        t = _decode_state(c, cfg)
    elif c["kind"] == "summary":
        t = _summary_state(c, cfg)
    else:
        t = _prefill_state(c, cfg)
    t["case"] = c
    return t


def run(t):
    c = t["case"]
    kind, K, W = c["kind"], c["K"], c["W"]
    if kind == "decode":
        return hils.hils_decode(t["q"], t["k"], t["v"], t["landmarks"], t["seq_lens"], S, K, t["out"], t["lse"], t["sel"],
                                bias=t["bias"], window=W, workspace=t["ws"])
    if kind == "decode_paged":
        return hils.hils_decode_paged(t["q"], t["k"], t["v"], t["landmarks"], t["table"], t["seq_lens"], S, K,
                                      bias=t["bias"], window=W, out=t["out"], lse=t["lse"], sel_idx=t["sel"],
                                      workspace=t["ws"])
    if kind == "decode_multi":
        return hils.hils_decode_multi(t["q"], t["k"], t["v"], t["landmarks"], t["seq_lens"], S, K, bias=t["bias"],
                                      window=W, out=t["out"], lse=t["lse"], sel_idx=t["sel"])
    if kind == "prefill":
        return hils.hils_prefill(t["q"], t["k"], t["v"], t["landmarks"], S, K, bias=t["bias"], window=W,
                                 workspace=t["ws"])
    if kind == "prefill_at":
        return hils.hils_prefill_at(t["q"], t["k"], t["v"], t["landmarks"], S, K, c["pos0"], bias=t["bias"], window=W)
    if kind == "train":
        out, lse, sel = hils.hils_attention(t["q"], t["k"], t["v"], t["landmarks"], S, K, bias=t["bias"], window=W)
        leaves = [t[n] for n in ("q", "k", "v", "landmarks", "bias") if t[n] is not None]
        return (out.detach(), lse, sel) + torch.autograd.grad(out, leaves, t["dout"])
    return hils.hils_landmark_summary(t["lq"], t["k"], S, seq_lens=t["lens"], landmarks=t["landmarks"], bias=t["bias"])


# --------------------------------------------------------------------------------------------------- work and tolerance
def work(case):
    c = dict(_DEFAULTS, **case)
    B, Hq, Hkv, d, K, W, M, T = (c[n] for n in ("B", "Hq", "Hkv", "d", "K", "W", "M", "T"))
    e = 4 if c["dtype"] == "f32" else 2
    C = _chunks(c)
    if c["kind"] == "summary":
        tokens = sum(min(n, C * S) for n in _lengths(c))
        rows = sum(min(C, (n + S - 1) // S) for n in _lengths(c))
        return {"bytes": Hkv * (tokens * d * e + rows * (2 * d * e + 4)), "flops": 4.0 * d * Hkv * tokens}
    if c["kind"].startswith("decode"):
        n = np.asarray(_lengths(c), dtype=np.int64)
        left = _left(n - 1, W)
        cand = left // S
        local = n - left
        picked = np.minimum(K, cand)
        # draft tokens of a sequence share 87 % of their chunks: what M of them have to load between them
        distinct = np.minimum(cand, picked * (1.0 + 0.13 * (M - 1)))
        b = Hkv * (float(cand.sum()) * (d * e + (4 if c["bias"] else 0)) + float((distinct * S + local).sum()) * 2 * d * e)
        b += B * M * (2.0 * Hq * d * e + 4 * Hq + 4 * Hkv * K)
        f = Hq * M * d * (2.0 * float(cand.sum()) + 4.0 * float((picked * S + local).sum()))
        return {"bytes": b, "flops": f}
    pos = _positions(c)
    left = _left(pos, W)
    cand = (left // S).astype(np.float64)
    attended = float((np.minimum(K, cand) * S + (pos - left) + 1).sum())
    rows, visible = len(pos), int(pos[-1]) + 1
    gathered, scoring = 4.0 * d * Hq * B * attended, 2.0 * d * Hq * B * float(cand.sum())
    kv, lm = B * Hkv * visible * d, B * Hkv * (visible // S) * (d * e + (4 if c["bias"] else 0))
    io = B * rows * (2.0 * Hq * d * e + 4 * Hq + 4 * Hkv * K)
    b, f = 2 * kv * e + lm + io, gathered + scoring
    if c["kind"] == "train":                              # dout in, dq, dk, dv, dlandmarks, dbias out; five products
        b += B * rows * 2.0 * Hq * d * e + 2 * kv * e + lm + 2 * kv * e + lm + io
        f += 2.5 * gathered
    return {"bytes": b, "flops": f}


def tolerance(case):
    c = dict(_DEFAULTS, **case)
    if c["dtype"] == "f32":
        return {"rel": 1e-5, "max": 1e-3, "differ": 1e-3}
    # bf16 results (gradients are sums of bf16 products); a group score that ties to the last fp32 bits may order two
    # chunks the other way
    return {"rel": 1e-2, "max": 0.6, "differ": 2e-3}

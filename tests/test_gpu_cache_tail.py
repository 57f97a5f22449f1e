"""Rows of a cache past a sequence's last token are never part of a result, whatever they hold (a cache that was allocated
and not filled holds any bits): the calls below on caches whose tails are NaN or infinite, against the CPU oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2607_02980_b200 as hils
from paper_2607_02980_b200 import workloads as wl
from parity import TOL_LSE, TOL_OUT

pytestmark = pytest.mark.gpu
DEV = "cuda"


def poison(inp, lens, value):
    for b, n in enumerate(lens):
        inp["k"][b, :, n:] = value
        inp["v"][b, :, n:] = value
        inp["landmarks"][b, :, n // 64:] = value


def check(got, ref, K, dtype="bf16"):
    """got: out [n, Hq, d], lse [n, Hq], sel [n, Hkv, K] of the rows of ref."""
    out, lse, sel = (t.float().cpu().numpy() if t.dtype != torch.int32 else t.cpu().numpy() for t in got)
    assert np.isfinite(out).all() and np.isfinite(lse).all()
    ok = (ref["margin"] >= 1e-3).all(axis=1)
    assert (sel[ok] == ref["sel_idx"][ok]).all()
    assert np.abs(out - ref["out"])[ok].max() <= TOL_OUT[dtype]
    assert np.abs(lse - ref["lse"])[ok].max() <= TOL_LSE[dtype]


@pytest.mark.parametrize("value", [float("nan"), float("inf"), 3e38])
@pytest.mark.parametrize("B,M,W,G", [(10, 4, 1, 4), (14, 3, 512, 4), (10, 4, 130, 3), (20, 2, 1, 8)])
def test_drafts_that_straddle_a_chunk(B, M, W, G, value):
    """The newest chunk is in the later tokens' windows only; the earlier tokens share the MMA tile with it (the batch is large
    enough for a sequence's tokens to be worked on together)."""
    cfg = wl.HilsConfig("tail", "decode", B, 8 * G, 8, 64 * 42, 128, 64, 16, "bf16", 700 + M, window=W)
    lens = [64 * (24 + b % 16) + (1 + b % (M - 1)) for b in range(B)]     # 1 .. M - 1 tokens past a boundary
    inp = wl.make_decode_inputs(cfg, "cpu", seq_lens=torch.tensor(lens, dtype=torch.int32))
    q = torch.randn((B, M, cfg.Hq, 128), generator=torch.Generator().manual_seed(B)).to(torch.bfloat16)
    poison(inp, lens, value)
    g = {n: t.to(DEV) for n, t in inp.items()}
    out, lse, sel = hils.hils_decode_multi(q.to(DEV), g["k"], g["v"], g["landmarks"], g["seq_lens"], 64, 16, window=W)
    torch.cuda.synchronize()
    for m in range(M):
        sl = torch.tensor([n - M + m + 1 for n in lens], dtype=torch.int32)
        ref = oracle.hils_decode(q[:, m].contiguous(), inp["k"], inp["v"], inp["landmarks"], None, sl, S=64, K=16, W=W)
        check((out[:, m], lse[:, m], sel[:, m]), ref, 16)


@pytest.mark.parametrize("dtype,impl,S,Hkv,pos0,L,W", [
    ("f32", "generic", 64, 1, 300, 200, 1),
    ("f32", "generic", 48, 2, 100, 333, 100),
    ("bf16", "generic", 64, 1, 300, 200, 1),
])
def test_slice_that_ends_inside_a_chunk(dtype, impl, S, Hkv, pos0, L, W):
    cfg = wl.HilsConfig("tail", "prefill", 2, 4 * Hkv, Hkv, (pos0 + L + 2 * S) // S * S, 128, S, 4, dtype, 730 + L, window=W)
    inp = wl.make_prefill_inputs(cfg, "cpu")
    n = pos0 + L
    assert n % S and cfg.L > n
    for t in (inp["k"], inp["v"]):
        t[:, :, n:] = float("nan")
    inp["landmarks"][:, :, n // S:] = float("nan")
    q = inp["q"][:, :, pos0:n].contiguous()
    g = {x: t.to(DEV) for x, t in inp.items()}
    out, lse, sel = hils.hils_prefill_at(q.to(DEV), g["k"], g["v"], g["landmarks"], S, 4, pos0, window=W, impl=impl)
    torch.cuda.synchronize()
    rows = np.arange(L)
    for b in range(2):
        ref = oracle.hils_rows(q, inp["k"], inp["v"], inp["landmarks"], None, S=S, K=4, W=W,
                               row_b=np.full(L, b, np.int32), row_qi=rows.astype(np.int32), row_pos=(pos0 + rows).astype(np.int64))
        check((out[b].transpose(0, 1), lse[b].T, sel[b].transpose(0, 1)), ref, 4, dtype)

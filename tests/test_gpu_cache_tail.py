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
    ("bf16", "fast", 64, 1, 300, 200, 1),              # query-major
    ("bf16", "fast", 64, 8, 3000, 1300, 512),          # chunk-major, local windows query-major
    ("bf16", "fast", 64, 1, 3000, 3300, 1),            # chunk-major
    ("bf16", "packed", 64, 1, 304, 200, 1),
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


@pytest.mark.parametrize("impl,L", [("fast", 900), ("fast", 3001), ("packed", 300), ("generic", 300)])
def test_a_sequence_is_not_spoilt_by_the_next_one(impl, L):
    """A tile of the first sequence's last chunk reaches into the rows of the second."""
    cfg = wl.HilsConfig("next", "prefill", 2, 4, 1, L, 128, 64, 16, "bf16", 760 + L)
    g = wl.make_prefill_inputs(cfg, DEV)
    run = lambda: hils.hils_prefill(g["q"], g["k"], g["v"], g["landmarks"], 64, 16, impl=impl)
    clean = run()
    for n in ("q", "k", "v"):
        g[n][1] = float("nan")
    got = run()
    torch.cuda.synchronize()
    for x, y in zip(got, clean):
        assert torch.equal(x[0], y[0])


@pytest.mark.parametrize("L", [300, 3001])
def test_gradients_of_a_sequence_that_ends_inside_a_chunk(L):
    """Caches longer than the sequence: the gradients are those of caches cut to it, and zero behind it."""
    cfg = wl.HilsConfig("tail", "prefill", 2, 8, 2, L, 128, 64, 8, "bf16", 780 + L)
    t = wl.make_prefill_inputs(cfg, DEV)
    dout = torch.randn(t["q"].shape, device=DEV, generator=torch.Generator(device=DEV).manual_seed(L)).to(torch.bfloat16)
    def grads(k, v):
        leaves = [x.clone().requires_grad_(True) for x in (t["q"], k, v, t["landmarks"])]
        out, lse, sel = hils.hils_attention(*leaves, 64, 8)
        return (out.detach(), lse.detach()) + torch.autograd.grad(out, leaves, dout)
    tail = torch.full((2, 2, 100, 128), float("nan"), dtype=torch.bfloat16, device=DEV)
    want = grads(t["k"], t["v"])
    got = grads(torch.cat([t["k"], tail], dim=2), torch.cat([t["v"], tail], dim=2))
    for i, (x, y) in enumerate(zip(got, want)):
        if i in (3, 4):                                        # dk, dv
            assert (x[:, :, L:] == 0).all()
            x = x[:, :, :L]
        # (sums in another order: the last bit of a bf16 gradient)
        assert (x.float() - y.float()).norm() <= 4e-3 * y.float().norm()


@pytest.mark.parametrize("K,impl,W,per_head,launches", [(16, "auto", 1, False, 1), (16, "auto", 200, False, 1), (8, "auto", 1, False, 3),
                                                        (16, "auto", 65, True, 3), (8, "generic", 65, False, 2)])
def test_decode_inside_a_chunk(K, impl, W, per_head, launches):
    cfg = wl.HilsConfig("tail", "decode", 3, 8, 2, 64 * 42, 128, 64, K, "bf16", 790 + K, window=W)
    lens = [64 * 41 + 1, 64 * 30 + 63, 17]
    inp = wl.make_decode_inputs(cfg, "cpu", seq_lens=torch.tensor(lens, dtype=torch.int32))
    if per_head:
        inp["landmarks"] = inp["landmarks"].repeat_interleave(4, dim=1).contiguous()
    poison(inp, lens, float("nan"))
    g = {n: t.to(DEV) for n, t in inp.items()}
    got = hils.hils_decode(g["q"], g["k"], g["v"], g["landmarks"], g["seq_lens"], 64, K, window=W, impl=impl)
    assert hils.last_launch_count() == launches
    torch.cuda.synchronize()
    check(got, oracle.hils_decode(inp["q"], inp["k"], inp["v"], inp["landmarks"], None, inp["seq_lens"], S=64, K=K, W=W), K)

"""A bias of minus infinity takes a chunk out of a sequence: it may still fill a place of the selection (where fewer than
top_k others are left: the lowest ids among equals, like any tie) and then has weight zero.  Every kernel that mixes chunks,
against the CPU oracle, with some, most and all chunks masked."""
import pytest
import torch

import paper_2607_02980_b200 as hils
from paper_2607_02980_b200 import workloads as wl
from parity import check_decode, check_prefill

pytestmark = pytest.mark.gpu
DEV = "cuda"


def masked_bias(cfg, share, heads=None, mask=float("-inf")):
    """bias [B, Hl, C] with `share` of the chunks masked, chunk 0 among them."""
    g = torch.Generator().manual_seed(cfg.seed)
    bias = torch.randn((cfg.B, heads or cfg.Hkv, cfg.C), generator=g)
    bias[torch.rand(bias.shape, generator=g) < share] = mask
    bias[:, :, 0] = mask
    return bias


def decode(cfg, share, seq=None, impl="auto", per_head=False, mask=float("-inf")):
    seq = torch.tensor(seq or [cfg.L - 97 * b for b in range(cfg.B)], dtype=torch.int32)
    inp = wl.make_decode_inputs(cfg, "cpu", seq_lens=seq)
    if per_head:
        inp["landmarks"] = inp["landmarks"].repeat_interleave(cfg.G, dim=1).contiguous()
    bias = masked_bias(cfg, share, cfg.Hq if per_head else None, mask)
    g = {n: t.to(DEV) for n, t in inp.items()}
    got = hils.hils_decode(g["q"], g["k"], g["v"], g["landmarks"], g["seq_lens"], 64, cfg.K, window=cfg.window,
                           bias=bias.to(DEV), impl=impl)
    torch.cuda.synchronize()
    check_decode(cfg, inp, *got, bias=bias, W=cfg.window)


def prefill(cfg, share, impl="auto", per_head=False, mask=float("-inf")):
    inp = wl.make_prefill_inputs(cfg, "cpu")
    if per_head:
        inp["landmarks"] = inp["landmarks"].repeat_interleave(cfg.G, dim=1).contiguous()
    bias = masked_bias(cfg, share, cfg.Hq if per_head else None, mask)
    g = {n: t.to(DEV) for n, t in inp.items()}
    got = hils.hils_prefill(g["q"], g["k"], g["v"], g["landmarks"], 64, cfg.K, bias=bias.to(DEV), window=cfg.window, impl=impl)
    torch.cuda.synchronize()
    check_prefill(cfg, inp, *got, bias=bias, W=cfg.window)


@pytest.mark.parametrize("share", [0.5, 0.97, 1.0])
@pytest.mark.parametrize("B,Hkv,T,K,W", [
    (2, 2, 64 * 20, 16, 1),            # every token takes nearly all its candidates
    (3, 2, 64 * 130, 16, 65),          # every candidate is ranked
    (2, 8, 64 * 400, 32, 512),         # lists longer than what is ranked
    (40, 8, 64 * 70, 16, 1),           # two CTAs per SM
])
def test_decode_in_clusters(B, Hkv, T, K, W, share):
    cfg = wl.HilsConfig("masked", "decode", B, 4 * Hkv, Hkv, T, 128, 64, K, "bf16", 1100 + B + K, window=W)
    decode(cfg, share)


@pytest.mark.parametrize("share", [0.5, 1.0])
def test_draft_tokens(share):
    B, M = 10, 4
    cfg = wl.HilsConfig("masked", "decode", B, 32, 8, 64 * 40, 128, 64, 16, "bf16", 1150)
    seq = torch.tensor([cfg.L - 61 * b for b in range(B)], dtype=torch.int32)
    inp = wl.make_decode_inputs(cfg, "cpu", seq_lens=seq)
    q = torch.randn((B, M, 32, 128), generator=torch.Generator().manual_seed(5)).to(torch.bfloat16)
    bias = masked_bias(cfg, share)
    g = {n: t.to(DEV) for n, t in inp.items()}
    out, lse, sel = hils.hils_decode_multi(q.to(DEV), g["k"], g["v"], g["landmarks"], g["seq_lens"], 64, 16, bias=bias.to(DEV))
    torch.cuda.synchronize()
    for m in range(M):
        one = dict(inp, q=q[:, m].contiguous(), seq_lens=seq - (M - 1 - m))
        check_decode(cfg, one, out[:, m], lse[:, m], sel[:, m], bias=bias)


@pytest.mark.parametrize("share", [0.5, 0.97, 1.0])
@pytest.mark.parametrize("T,K,W,per_head", [(64 * 40, 8, 1, False), (64 * 60, 16, 65, True)])
def test_decode_in_three_kernels(T, K, W, per_head, share):
    cfg = wl.HilsConfig("masked", "decode", 2, 8, 2, T, 128, 64, K, "bf16", 1155 + K, window=W)
    decode(cfg, share, per_head=per_head)
    assert hils.last_launch_count() == 3


@pytest.mark.parametrize("share", [0.5, 1.0])
@pytest.mark.parametrize("mode,dtype,d,L,K,W", [
    ("decode", "bf16", 128, 64 * 40, 16, 65),
    ("decode", "f32", 64, 64 * 30, 4, 1),
    ("prefill", "bf16", 128, 700, 4, 1),
    ("prefill", "f32", 96, 500, 4, 65),        # the row kernel
    ("prefill", "f32", 64, 700, 4, 1),         # the chunk-major kernels
])
def test_generic_kernels(mode, dtype, d, L, K, W, share):
    cfg = wl.HilsConfig("masked", mode, 2, 8, 2, L, d, 64, K, dtype, 1160 + d, window=W)
    (decode if mode == "decode" else prefill)(cfg, share, impl="generic")


@pytest.mark.parametrize("share", [0.5, 1.0])
def test_query_major_prefill(share):
    """No more candidates than top_k: one launch, chunk 0 first in every token's walk."""
    cfg = wl.HilsConfig("masked", "prefill", 3, 8, 2, 1000, 128, 64, 16, "bf16", 1170)
    prefill(cfg, share)
    assert hils.last_launch_count() == 1


@pytest.mark.parametrize("share", [0.5, 0.97, 1.0])
@pytest.mark.parametrize("B,Hkv,L,K,W,impl,per_head", [
    (1, 1, 3000, 5, 130, "auto", False),       # everything chunk-major
    (2, 2, 64 * 40 + 1, 16, 1, "auto", False),
    (1, 2, 64 * 50, 32, 1, "auto", True),
    (1, 2, 64 * 60, 40, 65, "auto", False),    # the selection kernel of top_k > 32
    (1, 2, 64 * 30, 8, 1, "packed", False),
])
def test_selected_prefill(B, Hkv, L, K, W, impl, per_head, share):
    cfg = wl.HilsConfig("masked", "prefill", B, 4 * Hkv, Hkv, L, 128, 64, K, "bf16", 1180 + K, window=W)
    prefill(cfg, share, impl=impl, per_head=per_head)


@pytest.mark.parametrize("L,K", [(64 * 60 + 9, 16), (64 * 60, 32), (64 * 60, 40)])
def test_a_query_that_is_not_a_number_spoils_its_own_row_only(L, K):
    """Its scores beat no threshold either: the selection still has to be K chunks that exist."""
    cfg = wl.HilsConfig("nan", "prefill", 1, 4, 1, L, 128, 64, K, "bf16", 1190 + K)
    g = wl.make_prefill_inputs(cfg, DEV)
    clean = hils.hils_prefill(g["q"], g["k"], g["v"], g["landmarks"], 64, K)
    rows = torch.tensor([0, 77, 64 * 50 + 3, L - 1], device=DEV)
    g["q"][:, :, rows] = float("nan")
    out, lse, sel = hils.hils_prefill(g["q"], g["k"], g["v"], g["landmarks"], 64, K)
    torch.cuda.synchronize()
    rest = torch.ones(L, dtype=torch.bool, device=DEV)
    rest[rows] = False
    assert torch.equal(out[:, :, rest], clean[0][:, :, rest]) and torch.equal(lse[:, :, rest], clean[1][:, :, rest])
    assert torch.isnan(out[:, :, rows]).all()
    for r in rows.tolist():
        ids = sel[0, 0, r].tolist()
        n = min(K, r // 64)
        assert ids[n:] == [-1] * (K - n) and sorted(set(ids[:n])) == ids[:n] and all(0 <= c < r // 64 for c in ids[:n])


@pytest.mark.parametrize("share", [0.5, 0.97])
@pytest.mark.parametrize("mode,L,K,impl", [("decode", 64 * 400, 32, "auto"), ("decode", 64 * 40, 8, "auto"), ("decode", 64 * 40, 8, "generic"),
                                           ("prefill", 1000, 16, "auto"), ("prefill", 3000, 5, "auto"), ("prefill", 64 * 60, 40, "auto")])
def test_masks_of_the_lowest_finite_number(mode, L, K, impl, share):
    cfg = wl.HilsConfig("lowest", mode, 1, 8, 2, L, 128, 64, K, "bf16", 1400 + K)
    (decode if mode == "decode" else prefill)(cfg, share, impl=impl, mask=torch.finfo(torch.float32).min)


def test_masks_of_the_lowest_finite_number_take_the_short_path():
    """A list with such masks has a histogram like any other (up to 256 of its chunks are ranked), where its span of 3.4e38 must not
    turn the bins' width into nothing: the kernel takes as long as with masks of -1e30.  (Without a histogram the radix selection
    over the cluster takes a quarter more.)"""
    B, T, K = 8, 64 * 400, 16
    cfg = wl.HilsConfig("path", "decode", B, 32, 8, T, 128, 64, K, "bf16", 1450)
    t = wl.make_decode_inputs(cfg, DEV)
    masked = torch.rand((B, 8, cfg.C), generator=torch.Generator().manual_seed(7)) < 0.7
    lowest = [torch.where(masked, m, torch.zeros(())).contiguous().to(DEV) for m in (-1e30, torch.finfo(torch.float32).min)]
    times, sels = ([], []), []
    hils.trace_enable(True)
    try:
        for i in range(60):
            got = hils.hils_decode(t["q"], t["k"], t["v"], t["landmarks"], t["seq_lens"], 64, K, bias=lowest[i & 1])
            (name, ms), = hils.trace_read()
            times[i & 1].append(ms)
            sels.append(got[2])
    finally:
        hils.trace_enable(False)
    assert name == "decode_cluster" and torch.equal(sels[0], sels[1])
    assert min(times[1]) <= 1.1 * min(times[0]), (min(times[0]), min(times[1]))

"""The one-launch decode kernel (clusters per (sequence, KV head)) against the CPU oracle at the sizes where
it can go wrong: candidate lists around its tiles of 64, around the switch from ranking every candidate to the
histogram, lists that agree in every score (the exact radix selection), ragged and invalid lengths, windows, every
column packing, draft tokens apart and grouped, pages out of range."""
import numpy as np
import pytest
import torch

import oracle
import paper_2607_02980_b200 as hils
from paper_2607_02980_b200 import workloads as wl
from parity import TOL_LSE, TOL_OUT, check_decode

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("B,T,seq,K,W,G,marks", [
    (3, 64 * 130, [64 * 17 + 1, 64 * 129, 64 * 130], 16, 1, 4, "random"),     # 17, 128 and 129 candidates
    (2, 64 * 70, [64 * 70, 64 * 65 + 1], 64, 65, 8, "random"),                # lists a little longer than K
    (1, 64 * 194, [64 * 192 + 1], 16, 1, 4, "random"),                        # 192 candidates, every CTA ranks them all
    (1, 64 * 194, [64 * 193 + 1], 16, 1, 8, "random"),                        # 193
    (1, 64 * 190, [64 * 190], 32, 1, 3, "equal"),                             # ties among all of them
    (40, 64 * 100, [64 * 100 - 61 * b for b in range(40)], 16, 1, 4, "three values"),    # three warps: 96 candidates, fewer and more
    (2, 64 * 400, [64 * 400, 64 * 260 + 7], 128, 512, 2, "random"),
    (2, 64 * 300, [64 * 300, 64 * 200], 16, 1, 4, "equal"),                   # every score ties: lowest ids
    (2, 64 * 300, [64 * 300 - 1, 5], 20, 130, 3, "three values"),
    (40, 64 * 150, None, 32, 1, 4, "three values"),                           # two CTAs per SM
    (1, 64 * 150, [64 * 150], 16, 1, 1, "random"),
    (2, 64 * 150, [64 * 150, 64 * 3], 1, 1, 5, "random"),
])
def test_against_the_oracle(B, T, seq, K, W, G, marks):
    Hkv = 2 if B < 40 else 8
    cfg = wl.HilsConfig("cluster", "decode", B, G * Hkv, Hkv, T, 128, 64, K, "bf16", 900 + K + B, n_needles=2, window=W)
    seq = seq or [T - 211 * b for b in range(B)]
    inp = wl.make_decode_inputs(cfg, "cpu", seq_lens=torch.tensor(seq, dtype=torch.int32))
    if marks == "equal":
        inp["landmarks"][:] = inp["landmarks"][:1, :1, :1].clone()
    elif marks == "three values":
        which = torch.randint(0, 3, (cfg.C,), generator=torch.Generator().manual_seed(3))
        inp["landmarks"] = inp["landmarks"][:, :, which].contiguous()
    bias = None if marks != "random" else wl.make_bias(cfg, "cpu")
    g = {n: t.to(DEV) for n, t in inp.items()}
    out, lse, sel = hils.hils_decode(g["q"], g["k"], g["v"], g["landmarks"], g["seq_lens"], 64, K, window=W,
                                     bias=None if bias is None else bias.to(DEV))
    torch.cuda.synchronize()
    assert hils.last_launch_count() == 1
    check_decode(cfg, inp, out, lse, sel, bias=bias, W=W)
    if marks == "equal":
        assert (sel.cpu() == torch.arange(K, dtype=torch.int32)).all()


@pytest.mark.parametrize("B,M,W,Hkv", [(2, 3, 1, 4), (10, 4, 200, 8), (5, 7, 512, 8)])
def test_draft_tokens_equal_single_calls_and_the_oracle(B, M, W, Hkv):
    cfg = wl.HilsConfig("drafts", "decode", B, 4 * Hkv, Hkv, 64 * 80 + 3, 128, 64, 16, "bf16", 950 + M, window=W)
    seq = [cfg.L - 331 * b for b in range(B)]
    seq[1] = 64 * 40 + 1                                     # the tokens see different numbers of chunks
    inp = wl.make_decode_inputs(cfg, "cpu", seq_lens=torch.tensor(seq, dtype=torch.int32))
    q = inp["q"][:, None].float() + 0.3 * torch.randn((B, M, cfg.Hq, 128), generator=torch.Generator().manual_seed(M))
    q = q.to(torch.bfloat16)
    bias = wl.make_bias(cfg, "cpu")
    g = {n: t.to(DEV) for n, t in inp.items()}
    out, lse, sel = hils.hils_decode_multi(q.to(DEV), g["k"], g["v"], g["landmarks"], g["seq_lens"], 64, 16,
                                           bias=bias.to(DEV), window=W)
    torch.cuda.synchronize()
    assert hils.last_launch_count() == 1
    for m in range(M):
        sl = torch.tensor([n - M + m + 1 for n in seq], dtype=torch.int32)
        o1, l1, s1 = hils.hils_decode(q[:, m].contiguous().to(DEV), g["k"], g["v"], g["landmarks"], sl.to(DEV), 64, 16,
                                      bias=bias.to(DEV), window=W)
        torch.cuda.synchronize()
        assert torch.equal(s1, sel[:, m])
        assert (o1.float() - out[:, m].float()).abs().max() <= 1.6e-2 and (l1 - lse[:, m]).abs().max() <= 1e-4
        ref = oracle.hils_decode(q[:, m], inp["k"], inp["v"], inp["landmarks"], bias, sl, S=64, K=16, W=W)
        ok = np.repeat(ref["margin"] >= 1e-3, 4, axis=1)
        assert np.abs(out[:, m].float().cpu().numpy() - ref["out"])[ok].max() <= TOL_OUT["bf16"]
        assert np.abs(lse[:, m].cpu().numpy() - ref["lse"])[ok].max() <= TOL_LSE["bf16"]


def test_invalid_lengths_and_pages_set_the_status_and_leave_the_rest_alone():
    cfg = wl.HilsConfig("bad", "decode", 3, 8, 2, 64 * 40, 128, 64, 16, "bf16", 970)
    inp = wl.make_decode_inputs(cfg, "cpu", seq_lens=torch.tensor([64 * 40, 64 * 20 + 9, 777], dtype=torch.int32))
    g = {n: t.to(DEV) for n, t in inp.items()}
    good = hils.hils_decode(g["q"], g["k"], g["v"], g["landmarks"], g["seq_lens"], 64, 16)
    p = hils.make_params(B=3, Hq=8, Hkv=2, Hl=2, L=0, T_max=cfg.L, C=cfg.C, d=128, chunk_size=64, top_k=16, dtype=1)
    ws = hils.alloc_workspace(p, True, DEV)
    lens = g["seq_lens"].clone()
    lens[1] = cfg.L + 1
    out, lse, sel = hils.hils_decode(g["q"], g["k"], g["v"], g["landmarks"], lens, 64, 16, workspace=ws)
    assert hils.poll_status(ws) == -7
    assert (out[1] == 0).all() and (lse[1] == 0).all() and (sel[1] == -1).all()
    for b in (0, 2):
        assert torch.equal(out[b], good[0][b]) and torch.equal(sel[b], good[2][b])
    from test_gpu_paged import paginate
    kp, vp, table = paginate(inp, cfg, 3)
    table[0, 39] = kp.shape[0]                                # the last token's own chunk of sequence 0
    ws[:256].zero_()
    out, lse, sel = hils.hils_decode_paged(g["q"], kp.to(DEV), vp.to(DEV), g["landmarks"], table.to(DEV), g["seq_lens"],
                                           64, 16, workspace=ws)
    assert hils.poll_status(ws) == -7
    assert torch.equal(sel, good[2]) and torch.equal(out[1:], good[0][1:])


@pytest.mark.parametrize("n,K,W", [(258, 32, 1), (300, 32, 1), (321, 64, 1), (449, 32, 1), (330, 16, 512), (150, 128, 1), (129, 127, 1)])
def test_lists_that_leave_some_ctas_few_candidates_or_none(n, K, W):
    """One sequence: eight CTAs per KV head, fewer full tiles of 64 candidates than that."""
    T = 64 * (n + (W + 62) // 64) + 5
    cfg = wl.HilsConfig("few", "decode", 1, 32, 8, T, 128, 64, K, "bf16", 980 + n, n_needles=2, window=W)
    inp = wl.make_decode_inputs(cfg, "cpu")
    g = {x: t.to(DEV) for x, t in inp.items()}
    got = hils.hils_decode(g["q"], g["k"], g["v"], g["landmarks"], g["seq_lens"], 64, K, window=W)
    torch.cuda.synchronize()
    check_decode(cfg, inp, *got, W=W)


def form(cfg, M=1):
    p = hils.make_params(B=cfg.B, Hq=cfg.Hq, Hkv=cfg.Hkv, Hl=cfg.Hkv, L=0, T_max=cfg.L, C=cfg.C, d=128, chunk_size=64, top_k=cfg.K,
                         window=cfg.window, dtype=1)
    return hils.call_form(p, True, M)[:3]


# want: tokens per unit, warps per CTA (no room for clusters of more than one)
@pytest.mark.parametrize("B,M,K,T,want", [(16, 3, 17, 64 * 90, (3, 6)), (32, 3, 16, 64 * 90, (3, 6)), (20, 4, 16, 64 * 90, (4, 6)),
                                          (40, 2, 33, 64 * 90, (2, 6)), (32, 4, 12, 64 * 65, (4, 3)), (40, 3, 8, 64 * 65, (3, 3)),
                                          (64, 2, 14, 64 * 65, (2, 3))])
def test_groups_of_draft_tokens_on_six_and_on_three_warps(B, M, K, T, want):
    """A group's tokens share the selection's warps (max(1, warps / tokens) each); the chunks are attended in the order of their
    scores and reported in ascending order."""
    cfg = wl.HilsConfig("groups", "decode", B, 32, 8, T, 128, 64, K, "bf16", 800 + M * B, n_needles=2, window=1)
    assert form(cfg, M) == want + (1,)
    lens = torch.tensor([T - (b * 371) % (T - 640) for b in range(B)], dtype=torch.int32)
    t = wl.make_decode_inputs(cfg, DEV, seq_lens=lens.to(DEV))
    q = torch.randn((B, M, 32, 128), generator=torch.Generator().manual_seed(M)).to(torch.bfloat16).to(DEV)
    out, lse, sel = hils.hils_decode_multi(q, t["k"], t["v"], t["landmarks"], t["seq_lens"], 64, K)
    torch.cuda.synchronize()
    assert hils.last_launch_count() == 1
    for m in range(M):
        o, l, s = hils.hils_decode(q[:, m].contiguous(), t["k"], t["v"], t["landmarks"], t["seq_lens"] - (M - 1 - m), 64, K)
        torch.cuda.synchronize()
        assert torch.equal(s, sel[:, m])
        held = torch.where(s < 0, torch.iinfo(torch.int32).max, s)
        assert (held[..., 1:] >= held[..., :-1]).all()
        # (two roundings to bf16 of sums in different orders, outputs below 2: twice 2^-8 = 8e-3)
        assert (o.float() - out[:, m].float()).abs().max() <= 1.6e-2 and (l - lse[:, m]).abs().max() <= 1e-4


@pytest.mark.parametrize("T,W", [(64 * 150, 512), (64 * 12, 512)])
def test_pages_of_local_chunks_out_of_range(T, W):
    """A warp's first item is asked for by one lane ahead of the cluster's first barrier, and given up there where it has no page:
    with a list of candidates to score and without one, the other sequence's results stay the same."""
    from test_gpu_paged import paginate
    cfg = wl.HilsConfig("gone", "decode", 2, 8, 2, T, 128, 64, 16, "bf16", 971, window=W)
    inp = wl.make_decode_inputs(cfg, "cpu", seq_lens=torch.tensor([T, T - 9], dtype=torch.int32))
    kp, vp, table = paginate(inp, cfg, 2)
    p = hils.make_params(B=2, Hq=8, Hkv=2, Hl=2, L=0, T_max=T, C=cfg.C, d=128, chunk_size=64, top_k=16, window=W, dtype=1)
    ws = hils.alloc_workspace(p, True, DEV)
    run = lambda: hils.hils_decode_paged(inp["q"].to(DEV), kp.to(DEV), vp.to(DEV), inp["landmarks"].to(DEV), table.to(DEV),
                                         inp["seq_lens"].to(DEV), 64, 16, window=W, workspace=ws)
    good = run()
    assert hils.poll_status(ws) == 0 and hils.last_launch_count() == 1
    table[0, T // 64 - 8:] = -1                                # (every chunk of the window but its oldest)
    out, lse, sel = run()
    assert hils.poll_status(ws) == -7
    assert torch.equal(sel, good[2]) and torch.equal(out[1], good[0][1]) and torch.equal(lse[1], good[1][1])


@pytest.mark.parametrize("T,marks", [(64 * 70, "random"), (64 * 300 + 5, "random"), (64 * 300, "equal"), (64 * 12, "random")])
def test_groups_in_clusters(T, marks):
    """Groups of four drafts on two CTAs, whose shares of the output meet in what ranking, listing (and, with ties, the radix
    selection) leave: every candidate ranked, a list, a list of equal scores, nothing to select."""
    B, M, K, W = 8, 4, 16, 512
    cfg = wl.HilsConfig("pairs", "decode", B, 32, 8, T, 128, 64, K, "bf16", 960, n_needles=2, window=W)
    assert form(cfg, M) == (4, 6, 2)
    lens = torch.tensor([T - 17 * b for b in range(B)], dtype=torch.int32)
    t = wl.make_decode_inputs(cfg, DEV, seq_lens=lens.to(DEV))
    if marks == "equal":
        t["landmarks"][:] = t["landmarks"][:1, :1, :1].clone()
    bias = None if marks == "equal" else wl.make_bias(cfg, DEV)
    q = torch.randn((B, M, 32, 128), generator=torch.Generator().manual_seed(T)).to(torch.bfloat16).to(DEV)
    out, lse, sel = hils.hils_decode_multi(q, t["k"], t["v"], t["landmarks"], t["seq_lens"], 64, K, window=W, bias=bias)
    torch.cuda.synchronize()
    assert hils.last_launch_count() == 1
    for m in range(M):
        o, l, s = hils.hils_decode(q[:, m].contiguous(), t["k"], t["v"], t["landmarks"], t["seq_lens"] - (M - 1 - m), 64, K, window=W, bias=bias)
        torch.cuda.synchronize()
        assert torch.equal(s, sel[:, m])
        # (two roundings to bf16 of sums in different orders, outputs below 2: twice 2^-8 = 8e-3)
        assert (o.float() - out[:, m].float()).abs().max() <= 1.6e-2 and (l - lse[:, m]).abs().max() <= 1e-4


@pytest.mark.parametrize("B,M,chunks,K,want", [(10, 1, 6200, 32, (1, 6, 1)), (16, 4, 1000, 32, (4, 6, 1)), (32, 1, 1700, 16, (1, 3, 1))])
def test_lists_that_fill_a_cta(B, M, chunks, K, want):
    """Against the same sequences one by one (other splits of the lists); the caches are pages that the sequences share."""
    cfg = wl.HilsConfig("long", "decode", B, 32, 8, 64 * chunks, 128, 64, K, "bf16", 961)
    assert form(cfg, M) == want
    g = torch.Generator(device=DEV).manual_seed(chunks)
    rnd = lambda *shape: torch.randn(shape, device=DEV, generator=g).to(torch.bfloat16)
    q, kp, vp, lm = rnd(B, M, 32, 128), rnd(97, 8, 64, 128), rnd(97, 8, 64, 128), rnd(B, 8, chunks, 128)
    table = torch.randint(0, 97, (B, chunks), device=DEV, generator=g).to(torch.int32)
    lens = torch.tensor([64 * chunks - 131 * b for b in range(B)], dtype=torch.int32, device=DEV)
    out, lse, sel = hils.hils_decode_multi(q, kp, vp, lm, lens, 64, K, block_table=table)
    torch.cuda.synchronize()
    assert hils.last_launch_count() == 1
    for b in range(B):
        for m in range(M):
            o, l, s = hils.hils_decode_paged(q[b:b + 1, m].contiguous(), kp, vp, lm[b:b + 1], table[b:b + 1], lens[b:b + 1] - (M - 1 - m), 64, K)
            torch.cuda.synchronize()
            assert torch.equal(s[0], sel[b, m])
            assert (o[0].float() - out[b, m].float()).abs().max() <= 1.6e-2 and (l[0] - lse[b, m]).abs().max() <= 1e-4


def test_a_mean_of_chunks_is_rounded_once():
    """Keys and landmarks of zeros: the n chunks of a sequence and the one token behind them weigh 1 each, and the output is the sum
    of their values, exact in fp32, over n + 1.  The values make it lie half way between two bf16 numbers, where a quotient that is off
    in its last place rounds to the wrong one."""
    B, T, K = 32, 64 * 33, 32
    cfg = wl.HilsConfig("mean", "decode", B, 8, 2, T, 128, 64, K, "bf16", 972)
    zeros = lambda *shape: torch.zeros(shape, dtype=torch.bfloat16)
    v = torch.ones((B, 2, T, 128))
    tie = 2 * (torch.arange(128) % 80) + 1                    # the means: 1 + tie / 256, tie odd
    for b in range(B):
        n = b + 2                                             # chunks, the last one's single token among them
        # n tie / 256 in numbers of eight bits: even steps of 1 / 256 above one, any below
        left = n * tie
        if n % 2 == 1:
            v[b, :, 64 * (n - 1):] -= 1 / 256
            left = left + 1
        for c in range(n - n % 2):
            step = torch.round(left / (2 * (n - n % 2 - c))) * 2
            v[b, :, 64 * c:64 * (c + 1) if c < n - 1 else T] += step / 256
            left = left - step
        assert (left == 0).all()
    want = (1 + torch.where(tie % 4 == 1, tie - 1, tie + 1) / 256).expand(B, 8, 128)      # (ties to even)
    assert torch.equal(v, v.to(torch.bfloat16).float())
    lens = torch.tensor([64 * (b + 1) + 1 for b in range(B)], dtype=torch.int32, device=DEV)
    q = torch.randn((B, 8, 128), generator=torch.Generator().manual_seed(1)).to(torch.bfloat16)
    args = [x.to(DEV) for x in (zeros(B, 2, T, 128), v.to(torch.bfloat16), zeros(B, 2, T // 64, 128))]
    out, lse, sel = hils.hils_decode(q.to(DEV), *args, lens, 64, K)
    torch.cuda.synchronize()
    assert hils.last_launch_count() == 1
    assert torch.equal(out.float().cpu(), want)
    qm = torch.stack([q, q], 1).to(DEV)
    many = [x.repeat(3, 1, 1, 1) for x in args]
    out = hils.hils_decode_multi(qm.repeat(3, 1, 1, 1), *many, lens.repeat(3) , 64, K)[0]
    torch.cuda.synchronize()
    assert torch.equal(out[:, 1].float().cpu(), want.repeat(3, 1, 1))

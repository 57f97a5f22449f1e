"""hils_prefill where its tokens are split between the query-major and the chunk-major kernels, and where the chunk-major
walk changes: all tokens query-major with ragged last tiles, a split inside the sequence, slices, KV heads walked together and
one after the other, selection rows of odd length, a workspace whose plan depends on the split."""
import numpy as np
import pytest
import torch

import oracle
import paper_2607_02980_b200 as hils
from paper_2607_02980_b200 import workloads as wl
from parity import compare_rows, group_scores

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,Hkv,L,K,W,bias_scale,pos0", [
    (1, 1, 65, 4, 1, 0.0, 0),          # one unit, one token past a chunk
    (3, 1, 129, 16, 1, 0.5, 0),        # every token takes all its candidates: one launch writes the selection
    (2, 2, 1000, 8, 65, 0.0, 0),       # query-major to the end of a ragged tile
    (16, 4, 2500, 8, 1, 60.0, 0),      # split; logits that raise the running reference and hide chunks
    (4, 8, 2500, 5, 130, 0.5, 0),      # split; selection rows of 20 bytes
    (2, 1, 3000, 5, 130, 0.5, 0),      # too few KV heads to split
    (2, 4, 5000, 4, 512, 0.5, 0),      # the others' local windows query-major too
    (1, 8, 2100, 8, 512, 0.5, 9001),   # a slice at an odd position, windows query-major
    (2, 2, 6001, 5, 897, 0.0, 0),      # the widest window, a ragged last unit
    (1, 2, 4200, 16, 1, 0.0, 0),       # KV heads together
    (1, 1, 16384, 16, 1, 0.0, 0),      # one KV head at a time, several query blocks' worth of lists
    (4, 8, 1500, 8, 64, 0.5, 300),     # a slice that begins among the query-major tokens
    (1, 2, 900, 8, 1, 0.0, 7777),      # a slice past them
])
def test_against_the_oracle_and_the_generic_kernels(B, Hkv, L, K, W, bias_scale, pos0):
    gen = torch.Generator(device="cuda").manual_seed(L + K)
    T = pos0 + L
    rnd = lambda h, n: torch.randn((B, h, n, 128), device="cuda", generator=gen).to(torch.bfloat16)
    q, k, v, lm = rnd(4 * Hkv, L), rnd(Hkv, T), rnd(Hkv, T), rnd(Hkv, T // 64)
    bias = torch.randn((B, Hkv, T // 64), device="cuda", generator=gen) * bias_scale if bias_scale else None
    run = lambda impl: (hils.hils_prefill_at(q, k, v, lm, 64, K, pos0, bias=bias, window=W, impl=impl) if pos0 else
                        hils.hils_prefill(q, k, v, lm, 64, K, bias=bias, window=W, impl=impl))
    (o1, l1, s1), (o2, l2, s2) = run("fast"), run("generic")
    torch.cuda.synchronize()
    # every row against the generic kernels where both select the same chunks (each is within 1e-3 of the oracle in lse, and
    # within 2e-2 in out before it is rounded)
    same = (s1 == s2).all(dim=-1).repeat_interleave(4, dim=1)       # (scores that tie in bf16 accumulation order may swap)
    assert same.float().mean().item() >= 0.99
    assert (o1.float() - o2.float()).abs().amax(dim=-1)[same].max().item() <= 3.2e-2
    assert (l1 - l2).abs()[same].max().item() <= 2e-3
    # the ends, the borders of units and tiles, and some more rows against the oracle, by its rules
    rows = np.unique(np.concatenate([np.arange(min(3, L)), np.arange(max(0, L - 3), L), np.arange(63, L, 512), np.arange(128, L, 640),
                                     np.random.default_rng(L).integers(0, L, 60)]))
    cpu = [x.cpu() for x in (q, k, v, lm)]
    for b in range(min(B, 2)):
        one = [x[b:b + 1] for x in cpu]
        bb = None if bias is None else bias[b:b + 1].cpu()
        def attend(rr, sel=None):
            n = len(rr)
            return oracle.hils_rows(*one, bb, S=64, K=K, W=W, row_b=np.zeros(n, np.int32), row_qi=rr.astype(np.int32),
                                    row_pos=(pos0 + rr).astype(np.int64), sel_idx=sel)
        pick = lambda x: x[b][:, rows].float().cpu().numpy().swapaxes(0, 1)
        compare_rows("bf16", K, 64, W, attend(rows), s1[b][:, rows].cpu().numpy().swapaxes(0, 1), pick(o1), pick(l1), pos0 + rows,
                     lambda idx, sel: attend(rows[idx], sel),
                     lambda r, nc: group_scores(one[0][0, :, int(rows[r])].float().numpy(), one[3][0].float().numpy(),
                                                None if bb is None else bb[0].numpy(), nc))


def test_workspace_covers_the_plan_without_the_query_major_tokens():
    """All tokens' partial outputs exceed what a call keeps at a time, those of the chunk-major tokens alone do not: the call
    then holds them all, and the reported size has to say so."""
    cfg = wl.HilsConfig("ws", "prefill", 1, 32, 8, 16384, 128, 64, 32, "bf16", 5, window=512)
    t = wl.make_prefill_inputs(cfg, "cuda")
    out, lse, sel = hils.hils_prefill(t["q"], t["k"], t["v"], t["landmarks"], 64, 32, window=512)
    launches = hils.last_launch_count()
    torch.cuda.synchronize()
    assert torch.isfinite(out).all() and torch.isfinite(lse).all()
    # (with less than the plan takes the call would fall back to smaller query blocks: more launches)
    p = hils.make_params(B=1, Hq=32, Hkv=8, Hl=8, L=16384, T_max=16384, C=256, d=128, chunk_size=64, top_k=32, window=512, dtype=1)
    ws = torch.zeros(2 * hils.workspace_bytes(p, False), dtype=torch.uint8, device="cuda")
    again = hils.hils_prefill(t["q"], t["k"], t["v"], t["landmarks"], 64, 32, window=512, workspace=ws)
    torch.cuda.synchronize()
    assert hils.last_launch_count() == launches
    assert torch.equal(again[0], out)

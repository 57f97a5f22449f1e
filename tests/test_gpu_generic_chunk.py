"""The fp32 chunk-major kernel in its forms (blocks of 128 tokens with all heads of a KV head; blocks of 64 or 32 tokens of one
head) against the CPU oracle: head counts that do not divide a warp's rows, blocks and chunks that end in the
middle of one another, an odd and an even number of blocks, slices, landmarks per query head, a routing query."""
import numpy as np
import pytest
import torch

import oracle
import paper_2607_02980_b200 as hils
from paper_2607_02980_b200 import workloads as wl
from parity import check_prefill, TOL_LSE, TOL_OUT

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("B,Hq,Hkv,L,d,S,K,W,bias,per_head", [
    (2, 4, 2, 1300, 128, 64, 4, 1, False, False),      # 64 tokens, 21 blocks, eight warps
    (2, 6, 2, 1217, 64, 48, 3, 100, True, True),       # 64 tokens, three heads, chunks of 48, per-head landmarks
    (4, 2, 2, 1281, 64, 64, 8, 65, True, False),       # 32 tokens, one head per KV head, 41 blocks
    (1, 3, 1, 230, 128, 64, 4, 70, True, True),        # 32 tokens, 8 blocks, eight warps
    (3, 4, 2, 1300, 128, 64, 4, 1, True, False),       # 128 tokens, all heads, 11 blocks, eight warps
    (3, 6, 2, 1217, 64, 16, 5, 1, True, True),         # 128 tokens, three heads, chunks of 16, four warps
    (1, 2, 1, 31, 64, 16, 2, 1, False, False),
    (1, 1, 1, 1612, 64, 64, 8, 1, False, False),       # 32 tokens, 51 blocks from the middle on
    (1, 1, 1, 1730, 64, 48, 8, 40, True, False),       # 55 from the ends on
    (1, 2, 1, 1000, 64, 64, 8, 130, True, False),      # 32 from the middle on
])
def test_against_the_oracle(B, Hq, Hkv, L, d, S, K, W, bias, per_head):
    cfg = wl.HilsConfig("fp32", "prefill", B, Hq, Hkv, L, d, S, K, "f32", 900 + L, window=W)
    inp = wl.make_prefill_inputs(cfg, "cpu")
    b = wl.make_bias(cfg, "cpu") if bias else None
    if per_head:
        g = torch.Generator().manual_seed(L)
        inp["landmarks"] = inp["landmarks"].repeat_interleave(Hq // Hkv, 1)
        inp["landmarks"] = inp["landmarks"] + 0.3 * torch.randn(inp["landmarks"].shape, generator=g)
        b = b.repeat_interleave(Hq // Hkv, 1).contiguous()
    g = {n: t.to(DEV) for n, t in inp.items()}
    out, lse, sel = hils.hils_prefill(g["q"], g["k"], g["v"], g["landmarks"], S, K, window=W, bias=None if b is None else b.to(DEV))
    torch.cuda.synchronize()
    assert hils.last_launch_count() == 3
    check_prefill(cfg, inp, out, lse, sel, bias=b, W=W)


def compare(inp, rows, out, lse, sel, **kw):
    """Attention against the oracle on the kernel's own selection, and that selection against the oracle's: two scores of at most
    0.1 in fp32 sums of 128 products differ by less than 1e-5 from their exact values' difference."""
    sel = sel.cpu().numpy().transpose(0, 2, 1, 3)
    t = (inp["q"], inp["k"], inp["v"], inp["landmarks"], None)
    res = oracle.hils_prefill(*t, S=64, K=4, W=1, rows=rows, **kw)
    ok = res["margin"] >= 1e-5
    assert ok.mean() > 0.9 and (sel[ok] == res["sel_idx"][ok]).all()
    res = oracle.hils_prefill(*t, S=64, K=4, W=1, rows=rows, sel_idx=np.ascontiguousarray(sel), **kw)
    assert np.abs(out.cpu().numpy().transpose(0, 2, 1, 3) - res["out"]).max() <= TOL_OUT["f32"]
    assert np.abs(lse.cpu().numpy().transpose(0, 2, 1) - res["lse"]).max() <= TOL_LSE["f32"]


@pytest.mark.parametrize("L,pos0,T", [(700, 933, 1700), (129, 64, 193)])
def test_slice(L, pos0, T):
    cfg = wl.HilsConfig("fp32", "prefill", 2, 4, 2, T, 64, 64, 4, "f32", 77)
    inp = wl.make_prefill_inputs(cfg, "cpu")
    got = hils.hils_prefill_at(inp["q"][:, :, pos0:pos0 + L].contiguous().to(DEV), *[inp[n].to(DEV) for n in ("k", "v", "landmarks")], 64, 4, pos0)
    torch.cuda.synchronize()
    compare(inp, np.arange(pos0, pos0 + L), *got)


@pytest.mark.parametrize("L", [260, 1500])
def test_routing_query(L):
    cfg = wl.HilsConfig("fp32", "prefill", 2, 4, 2, L, 128, 64, 4, "f32", 78)
    inp = wl.make_prefill_inputs(cfg, "cpu")
    qr = inp["q"] + 0.5 * torch.randn(inp["q"].shape, generator=torch.Generator().manual_seed(5))
    got = hils.hils_prefill(*[inp[n].to(DEV) for n in ("q", "k", "v", "landmarks")], 64, 4, q_route=qr.to(DEV))
    torch.cuda.synchronize()
    compare(inp, np.arange(L), *got, q_route=qr)

"""The tcgen05 backward where its walk changes: fewer entries than a tile, ragged last tiles, a sequence that ends inside a
chunk, KV heads walked together and one after the other, more than one query block, K above and at the tile's edges."""
import pytest
import torch

import paper_2607_02980_b200 as hils
from paper_2607_02980_b200 import workloads as wl

pytestmark = pytest.mark.gpu


# bf16 probabilities and d S on one side, fp32 on the other: relative to the largest entry of each gradient
@pytest.mark.parametrize("B,Hkv,L,K,W,with_bias", [
    (1, 1, 64, 1, 1, False),
    (1, 1, 97, 1, 1, True),
    (2, 2, 127, 3, 64, True),
    (3, 1, 1025, 33, 65, False),
    (1, 2, 4100, 16, 1, True),        # a KV head gives every CTA too few tiles: KV heads together
    (1, 2, 16384 + 129, 16, 1, True),  # one KV head at a time, and a second query block with few tiles
])
def test_against_the_generic_kernel(B, Hkv, L, K, W, with_bias):
    cfg = wl.HilsConfig("bwd", "prefill", B, 4 * Hkv, Hkv, L, 128, 64, K, "bf16", 300 + L)
    gen = torch.Generator(device="cuda").manual_seed(L)
    shape = lambda h, n: (B, h, n, 128)
    q, k, v, lm, dout = (torch.randn(shape(h, n), device="cuda", generator=gen).to(torch.bfloat16)
                         for h, n in ((cfg.Hq, L), (Hkv, L), (Hkv, L), (Hkv, cfg.C), (cfg.Hq, L)))
    bias = torch.randn((B, Hkv, cfg.C), device="cuda", generator=gen) if with_bias else None
    out, lse, sel = hils.hils_prefill(q, k, v, lm, 64, K, bias=bias, window=W)
    args = (q, k, v, lm, 64, K, out, lse, sel, dout)
    got = hils.hils_prefill_backward(*args, bias=bias, window=W, impl="fast")
    ref = hils.hils_prefill_backward(*args, bias=bias, window=W, impl="generic")
    torch.cuda.synchronize()
    for g, r, name in zip(got, ref, ("dq", "dk", "dv", "dlandmarks", "dbias")):
        if g is not None:
            assert torch.isfinite(g).all(), name
            assert (g - r).abs().max().item() <= 2e-2 * r.abs().max().item() + 1e-6, name

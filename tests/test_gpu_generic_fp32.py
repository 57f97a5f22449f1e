"""The fp32 chunk-major kernels and the generic row kernel against the CPU oracle at the edges of their tiles: chunk
sizes that do not fill 64 keys, a ragged last chunk, rows around a block of 128, wide windows, both head dimensions the
chunk-major kernels take, and one they leave to the row kernel; selections longer than one and two registers per lane."""
import pytest
import torch

import paper_2607_02980_b200 as hils
from paper_2607_02980_b200 import workloads as wl
from parity import check_prefill

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("B,Hq,Hkv,L,d,S,K,W,bias", [
    (1, 1, 1, 129, 64, 64, 2, 1, False),
    (2, 4, 2, 300, 128, 48, 3, 100, True),
    (1, 2, 1, 1000, 64, 16, 40, 17, True),          # more than 32 selected, a row of up to 42 slots
    (1, 1, 1, 700, 64, 5, 70, 1, False),            # more than 64 selected
    (1, 2, 2, 260, 96, 64, 2, 1, True),             # row kernel: d = 96
    (1, 2, 1, 400, 256, 100, 2, 130, False),        # row kernel: chunks of more than 64 tokens
    (1, 1, 1, 200, 32, 64, 4, 1, False),
])
def test_against_the_oracle(B, Hq, Hkv, L, d, S, K, W, bias):
    cfg = wl.HilsConfig("fp32", "prefill", B, Hq, Hkv, L, d, S, K, "f32", 500 + L, window=W)
    inp = wl.make_prefill_inputs(cfg, "cpu")
    b = wl.make_bias(cfg, "cpu") if bias else None
    g = {n: t.to(DEV) for n, t in inp.items()}
    out, lse, sel = hils.hils_prefill(g["q"], g["k"], g["v"], g["landmarks"], S, K, window=W, bias=None if b is None else b.to(DEV))
    torch.cuda.synchronize()
    check_prefill(cfg, inp, out, lse, sel, bias=b, W=W)

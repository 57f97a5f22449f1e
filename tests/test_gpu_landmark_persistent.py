"""hils_landmark_summary where a warp of the persistent kernel takes several chunks: more chunks than warps on the GPU,
lengths that leave some sequences empty and some chunks partial, one and eight landmark heads per KV head."""
import numpy as np
import pytest
import torch

import oracle
import paper_2607_02980_b200 as hils
from paper_2607_02980_b200 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,Hkv,per,L,seq", [
    (4, 4, 1, 64 * 400, [64 * 400, 64 * 13 + 1, 0, 64 * 399 - 5]),
    (2, 1, 8, 64 * 1300, [64 * 1300, 64 * 1100 + 63]),
])
def test_against_the_oracle(B, Hkv, per, L, seq):
    cfg = wl.HilsConfig("many", "decode", B, Hkv * per, Hkv, L, 128, 64, 16, "bf16", 70 + per)
    k = wl.make_decode_inputs(cfg, "cpu", seq_lens=torch.tensor(seq, dtype=torch.int32))["k"]
    lq = wl.make_landmark_queries(cfg, "cpu", Hl=Hkv * per)
    sl = torch.tensor(seq, dtype=torch.int32)
    lm, b = hils.hils_landmark_summary(lq.cuda(), k.cuda(), 64, seq_lens=sl.cuda())
    torch.cuda.synchronize()
    ref_lm, ref_b = oracle.hils_landmarks(lq, k, seq_lens=sl, S=64)
    assert np.abs(lm.float().cpu().numpy() - ref_lm).max() <= 2e-2
    assert np.abs(b.cpu().numpy() - ref_b).max() <= 2e-5

"""The query-major prefill's chunk lists where the selection rows of a call reach shared memory in both ways: 16-byte aligned rows
of full blocks by a bulk copy, the others by ordinary loads.  With an odd top_k and an odd length it is every fourth (sequence, KV
head) that is aligned, but for its ragged last block; a CTA walks many units of both kinds."""
import pytest
import torch

import paper_2607_02980_b200 as hils
import test_gpu_prefill_split as split

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,Hkv,L,K,W", [
    (4, 8, 1501, 17, 1),       # 768 units, 64 tokens' rows at a time
    (3, 8, 2477, 35, 1),       # 936 units, 32 tokens' rows at a time
    (5, 8, 1437, 15, 65),      # a row's share of the window
])
def test_rows_aligned_in_some_units_and_not_in_others(B, Hkv, L, K, W):
    aligned = {(4 * K * (pair * L + 64 * blk)) % 16 == 0 and (4 * K * min(64, L - 64 * blk)) % 16 == 0
               for pair in range(B * Hkv) for blk in range((L + 63) // 64)}
    assert aligned == {True, False}
    split.test_against_the_oracle_and_the_generic_kernels(B, Hkv, L, K, W, 0.5, 0)
    t = [torch.randn((B, h, n, 128), device="cuda").to(torch.bfloat16) for h, n in ((4 * Hkv, L), (Hkv, L), (Hkv, L), (Hkv, L // 64))]
    first = hils.hils_prefill(*t, 64, K, window=W)
    assert hils.last_launch_count() == 2                  # selection and this kernel
    for _ in range(5):                                    # (the same rows in the same order: the same bits)
        again = hils.hils_prefill(*t, 64, K, window=W)
        torch.cuda.synchronize()
        assert all(torch.equal(x, y) for x, y in zip(first, again))

"""Selection with equal scores: integer-valued queries and landmarks, whose products are exact whatever the order of the sum.
Equal scores go to the lower chunk id, also where more candidates tie at the K-th score than a buffer holds."""
import pytest
import torch

import paper_2607_02980_b200 as hils

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,K,high", [(2000, 4, 0), (2900, 16, 0), (2900, 17, 1), (5000, 32, 1), (5000, 16, 2), (6500, 31, 2)])
def test_selection_is_the_generic_kernels(L, K, high):
    gen = torch.Generator(device="cuda").manual_seed(L)
    ints = lambda h, n, lim: torch.randint(-lim, lim + 1, (2, h, n, 128), device="cuda", generator=gen).to(torch.bfloat16)
    q, lm = ints(8, L, high), ints(2, L // 64, high)
    lm[..., 4:] = 0                       # few distinct scores
    k, v = ints(2, L, 1), ints(2, L, 1)
    args = (q, k, v, lm, 64, K)
    s1, s2 = hils.hils_prefill(*args, impl="fast", window=65)[2], hils.hils_prefill(*args, impl="generic", window=65)[2]
    torch.cuda.synchronize()
    assert torch.equal(s1, s2)

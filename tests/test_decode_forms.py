"""The form that the plan of the one-launch decode kernel chooses, for calls that stand close to what its shared memory holds: long
candidate lists, groups of draft tokens, two CTAs per SM.  Host only: the plan asks the device for clusters alone, and none of
these calls has room for one of more than one CTA (148 SMs)."""
import pytest

import paper_2607_02980_b200 as hils


def form(B, M, Hkv, G, T, K, W):
    p = hils.make_params(B=B, Hq=G * Hkv, Hkv=Hkv, Hl=Hkv, L=0, T_max=T, C=T // 64, d=128, chunk_size=64, top_k=K, window=W, dtype=1)
    return hils.call_form(p, True, M)


@pytest.mark.parametrize("B,M,Hkv,G,T,K,W,want", [
    # one token, one CTA per SM: the list of 5900 candidates is a CTA's own
    (10, 1, 8, 4, 64 * 6200, 32, 1, (1, 6, 1)),
    (24, 1, 8, 8, 64 * 5900, 32, 1, (1, 6, 1)),
    (10, 4, 4, 8, 64 * 6250, 32, 512, (1, 6, 1)),
    # two CTAs per SM
    (32, 1, 8, 4, 64 * 1700, 16, 1, (1, 3, 1)),
    (40, 2, 2, 4, 64 * 1300, 128, 512, (1, 3, 1)),
    (16, 3, 4, 8, 64 * 1100, 128, 1, (1, 3, 1)),
    (40, 1, 8, 4, 64 * 1340, 16, 1, (1, 3, 1)),
    (40, 1, 8, 4, 64 * 1400, 16, 1, (1, 6, 1)),        # 320 units: two per SM would take two turns, one per SM takes three
    # draft tokens of a sequence share a unit, six warps
    (16, 4, 8, 4, 64 * 1000, 32, 1, (4, 6, 1)),
    (16, 3, 8, 4, 64 * 1024, 8, 1, (3, 6, 1)),
    (64, 4, 2, 4, 64 * 1000, 16, 1, (4, 6, 1)),
    (40, 3, 8, 4, 64 * 768, 8, 1, (3, 6, 1)),
    (40, 3, 8, 4, 64 * 1024, 8, 1, (1, 3, 1)),         # more groups than SMs: apart
    (64, 4, 4, 8, 64 * 800, 32, 1, (1, 3, 1)),
    # and two CTAs per SM, where the lists are short
    (32, 4, 8, 4, 64 * 65, 12, 1, (4, 3, 1)),
    (40, 2, 8, 8, 64 * 65, 8, 1, (2, 3, 1)),
])
def test_calls_that_fill_the_shared_memory(B, M, Hkv, G, T, K, W, want):
    assert form(B, M, Hkv, G, T, K, W)[:3] == want

"""hils_call_form on the host: errors, calls that neither kernel takes, and the forms of the fp32 chunk-major kernel and of the one-launch
decode kernel at the sizes that test_gpu_generic_chunk.py and test_gpu_decode_cluster.py compare with the oracle (148 SMs)."""
import ctypes

import pytest

import paper_2607_02980_b200 as hils


def params(B, Hq, Hkv, L, d, S, K, dtype, W=1, Hl=None, T=0):
    return hils.make_params(B=B, Hq=Hq, Hkv=Hkv, Hl=Hl or Hkv, L=L, T_max=T, C=(T or L) // S, d=d, chunk_size=S, top_k=K, window=W, dtype=dtype)


def test_errors_and_other_kernels():
    lib, form = hils.load_library(), (ctypes.c_int32 * 4)()
    p = params(1, 8, 2, 1000, 128, 64, 4, 0)
    assert lib.hils_call_form(None, 0, 1, form) == -1
    assert lib.hils_call_form(ctypes.byref(p), 0, 1, None) == -1
    assert lib.hils_call_form(ctypes.byref(p), 0, 0, form) == -1
    with pytest.raises(hils.HilsError):
        hils.call_form(params(1, 7, 2, 1000, 128, 64, 4, 0), False)
    assert hils.call_form(params(1, 8, 2, 4096, 128, 64, 16, 1), False) == (0, 0, 0, 0)             # bf16 prefill
    assert hils.call_form(params(1, 8, 2, 500, 96, 64, 4, 0), False) == (0, 0, 0, 0)                # the row kernel
    assert hils.call_form(params(1, 8, 2, 0, 128, 64, 8, 1, T=4096), True) == (0, 0, 0, 0)          # three launches
    assert hils.call_form(params(1, 8, 2, 0, 128, 64, 16, 1, Hl=8, T=4096), True) == (0, 0, 0, 0)   # a landmark per query head


@pytest.mark.parametrize("B,Hq,Hkv,L,d,S,K,W,want", [
    (2, 4, 2, 1300, 128, 64, 4, 1, (64, 1, 8, 0)),
    (2, 6, 2, 1217, 64, 48, 3, 100, (64, 1, 4, 0)),
    (4, 2, 2, 1281, 64, 64, 8, 65, (32, 1, 4, 0)),
    (1, 3, 1, 230, 128, 64, 4, 70, (32, 1, 8, 1)),
    (3, 4, 2, 1300, 128, 64, 4, 1, (128, 2, 8, 0)),
    (3, 6, 2, 1217, 64, 16, 5, 1, (128, 3, 4, 0)),
    (1, 2, 1, 31, 64, 16, 2, 1, (32, 1, 4, 1)),
    (1, 1, 1, 1612, 64, 64, 8, 1, (32, 1, 4, 1)),
    (1, 1, 1, 1730, 64, 48, 8, 40, (32, 1, 4, 0)),
    (1, 2, 1, 1000, 64, 64, 8, 130, (32, 1, 4, 1)),
])
def test_fp32_prefill(B, Hq, Hkv, L, d, S, K, W, want):
    assert hils.call_form(params(B, Hq, Hkv, L, d, S, K, 0, W=W), False) == want


@pytest.mark.parametrize("B,Hkv,T,K,W,G,want", [
    (40, 8, 64 * 100, 16, 1, 4, (1, 3, 1, 96)),
    (40, 8, 64 * 150, 32, 1, 4, (1, 3, 1, 96)),
    (16, 8, 64 * 150, 32, 1, 4, (1, 6, 1, 128)),
])
def test_decode(B, Hkv, T, K, W, G, want):
    assert hils.call_form(params(B, G * Hkv, Hkv, 0, 128, 64, K, 1, W=W, T=T), True) == want

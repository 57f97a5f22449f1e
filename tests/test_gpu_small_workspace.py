"""Prefill in workspaces smaller than the ones the size queries report (those are what the fastest kernels take): smaller query
blocks, or the row kernel in fp32, with the same results; refused without a launch where even those do not fit."""
import pytest
import torch

import paper_2607_02980_b200 as hils
from paper_2607_02980_b200 import workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda"


def reported(cfg):
    p = hils.make_params(B=cfg.B, Hq=cfg.Hq, Hkv=cfg.Hkv, Hl=cfg.Hkv, L=cfg.L, T_max=cfg.L, C=cfg.C, d=cfg.d, chunk_size=64,
                         top_k=cfg.K, window=cfg.window, dtype=0 if cfg.dtype == "f32" else 1)
    return p, hils.workspace_bytes(p, False)


@pytest.mark.parametrize("B,Hkv,L,K,W", [(1, 2, 20000, 16, 1), (2, 2, 17000, 8, 512), (1, 1, 9001, 40, 65)])
def test_query_blocks_shrink_to_the_workspace(B, Hkv, L, K, W):
    cfg = wl.HilsConfig("ws", "prefill", B, 4 * Hkv, Hkv, L, 128, 64, K, "bf16", 1300 + K, window=W)
    g = wl.make_prefill_inputs(cfg, DEV)
    run = lambda ws: hils.hils_prefill(g["q"], g["k"], g["v"], g["landmarks"], 64, K, window=W, workspace=ws)
    n = reported(cfg)[1]
    # partial outputs of 2048 tokens, the tails of their lists (as many again at most), the index of all tokens
    slots = K + (W + 62) // 64 + 1
    least = B * Hkv * slots * (2 * 2048 * 1100 + 24 * L) + 64 * 1024 * L // 64 + (1 << 20)
    assert least < n
    full = run(None)
    for size in (n - 4096, (n + least) // 2, least):
        ws = torch.full((n,), 255, dtype=torch.uint8, device=DEV)
        ws[:256].zero_()
        got = run(ws[:size])
        torch.cuda.synchronize()
        assert all(torch.equal(x, y) for x, y in zip(got, full))
        assert (ws[size:] == 255).all() and hils.poll_status(ws) == 0
    with pytest.raises(hils.HilsError):
        run(ws[:B * Hkv * K * 2048 * 1024])


def test_a_slice_stays_inside_the_workspace_it_was_given():
    cfg = wl.HilsConfig("ws", "prefill", 1, 8, 2, 12000, 128, 64, 16, "bf16", 1340)
    g = wl.make_prefill_inputs(cfg, DEV)
    n, q = reported(cfg)[1], g["q"][:, :, 2000:].contiguous()
    run = lambda ws: hils.hils_prefill_at(q, g["k"], g["v"], g["landmarks"], 64, 16, 2000, workspace=ws)
    full = run(None)
    ws = torch.full((n,), 255, dtype=torch.uint8, device=DEV)
    ws[:256].zero_()
    got = run(ws[:n // 2])
    torch.cuda.synchronize()
    assert all(torch.equal(x, y) for x, y in zip(got, full))
    assert (ws[n // 2:] == 255).all()
    with pytest.raises(hils.HilsError):
        run(ws[:n // 20])


def test_fp32_without_scratch_takes_the_row_kernel():
    cfg = wl.HilsConfig("ws", "prefill", 1, 2, 1, 1000, 64, 64, 4, "f32", 1350)
    g = wl.make_prefill_inputs(cfg, DEV)
    ws = torch.zeros(256, dtype=torch.uint8, device=DEV)
    a = hils.hils_prefill(g["q"], g["k"], g["v"], g["landmarks"], 64, 4)
    assert hils.last_launch_count() == 3
    b = hils.hils_prefill(g["q"], g["k"], g["v"], g["landmarks"], 64, 4, workspace=ws)
    assert hils.last_launch_count() == 2
    torch.cuda.synchronize()
    assert torch.equal(a[2], b[2]) and (a[0] - b[0]).abs().max() <= 1e-5 and (a[1] - b[1]).abs().max() <= 1e-5


def test_host_arena_smaller_than_reported():
    cfg = wl.HilsConfig("ws", "prefill", 1, 8, 2, 7000, 128, 64, 16, "bf16", 1360)
    p, n = reported(cfg)
    inp = {x: t.pin_memory() for x, t in wl.make_prefill_inputs(cfg, "cpu").items()}
    runner = hils.HostRunner(p, False, DEV)
    args = [inp[x] for x in ("q", "k", "v", "landmarks")]
    want = [t.clone() for t in (runner.run(*args), torch.cuda.synchronize())[0]]
    runner.arena = runner.arena[:runner.arena.numel() - n // 3]
    got = runner.run(*args)
    torch.cuda.synchronize()
    assert all(torch.equal(x, y) for x, y in zip(got, want))
    runner.arena = runner.arena[:runner.arena.numel() - n // 2]
    with pytest.raises(hils.HilsError):
        runner.run(*args)

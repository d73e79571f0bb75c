"""The give-up path of the kernels' bounded waits, exercised without a fault or a hang.

Every wait inside the tensor-core forward and backward, the paged decode and the segmented summary has a wall-clock limit.
Here the limit is set to a few milliseconds and a test hook withholds something a wait needs (the forward's last key tile;
the last query tile of the backward's dK/dV kernel, whose issuing warp polls two barriers in a loop of its own; the last
tile of a share of the paged decode; one segment's carried state, in global or in shared memory): the wait runs out, every role of the CTA drains, tensor memory is freed, the kernel RETURNS, and the
status word of the workspace reads MKA_ERR_TIMEOUT.  The next ordinary call on the same stream must then match the
oracle, which shows that the context and the library are still healthy.
"""
import ctypes

import numpy as np
import pytest
import torch

from gpu_helpers import check, np64, problem

pytestmark = pytest.mark.gpu
MKA_ERR_TIMEOUT = 7


@pytest.fixture(scope="module")
def mka():
    import paper_2603_20586_b200 as m
    assert torch.cuda.is_available()
    return m


@pytest.fixture()
def short_limit(mka):
    old = mka.mka_set_wait_limit_us(3000)
    yield 3000
    mka.mka_set_wait_limit_us(old)


@pytest.mark.parametrize("d", [128, 64])
def test_forward_wait_runs_out_and_the_next_call_is_correct(mka, orc, short_limit, d):
    B, H, T, W, N = 1, 2, 300, 96, (300, 300, 160)
    P = problem(91, B, H, T, d, N, 32, torch.bfloat16, router_std=0.3)
    gate = mka.mka_router(P["X"], P["W_r"], None)
    ws = mka.alloc_workspace(mka.make_shape(B, H, T, d, 32, W), N, mka.MKA_WS_FWD, "cuda")
    stalled = mka.make_shape(B, H, T, d, 32, W, flags=mka.MKA_FLAG_TEST_STALL)
    assert mka.mka_fwd_kernel_kind(stalled, P["K"], P["V"]) == 1
    t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    t0.record()
    mka.mka_fwd(stalled, P["Q"], P["K"], P["V"], gate, ws=ws)
    t1.record()
    assert mka.mka_device_status(ws) == MKA_ERR_TIMEOUT           # synchronises the stream: the kernel came back
    assert t0.elapsed_time(t1) < 1000.0                           # after about one limit, not after the one-second default
    # the same problem without the hook, same workspace, same stream
    shape = mka.make_shape(B, H, T, d, 32, W)
    O, LSE = mka.mka_fwd(shape, P["Q"], P["K"], P["V"], gate, ws=ws)
    assert mka.mka_device_status(ws) == 0
    rg, _ = orc.router(np64(P["X"]), np64(P["W_r"]))
    Or, Lr = orc.fwd(P["Q"], P["K"], P["V"], rg, W)
    check(O, Or, torch.bfloat16, "forward after a timed-out call")
    assert np.abs(np64(LSE) - Lr).max() <= 2e-3


@pytest.mark.parametrize("d", [128, 64])
def test_backward_wait_runs_out_and_the_next_call_is_correct(mka, orc, short_limit, d):
    B, H, T, W, N = 1, 2, 300, 96, (300, 300, 160)
    P = problem(93, B, H, T, d, N, 32, torch.bfloat16, router_std=0.3, with_dO=True)
    gate = mka.mka_router(P["X"], P["W_r"], None)
    shape = mka.make_shape(B, H, T, d, 32, W)
    O, LSE = mka.mka_fwd(shape, P["Q"], P["K"], P["V"], gate)
    assert mka.mka_bwd_kernel_kind(shape, P["K"], P["V"]) == 1
    ws = mka.alloc_workspace(shape, N, mka.MKA_WS_BWD, "cuda")
    stalled = mka.make_shape(B, H, T, d, 32, W, flags=mka.MKA_FLAG_TEST_STALL)
    t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    t0.record()
    mka.mka_bwd(stalled, P["Q"], P["K"], P["V"], gate, O, LSE, P["dO"], R=P["X"], ws=ws)
    t1.record()
    assert mka.mka_device_status(ws) == MKA_ERR_TIMEOUT
    assert t0.elapsed_time(t1) < 1000.0
    g = mka.mka_bwd(shape, P["Q"], P["K"], P["V"], gate, O, LSE, P["dO"], R=P["X"], ws=ws)
    assert mka.mka_device_status(ws) == 0
    rg, _ = orc.router(np64(P["X"]), np64(P["W_r"]))
    ref = orc.bwd(P["Q"], P["K"], P["V"], rg, P["dO"], W)
    check(g["dQ"], ref["dQ"], torch.bfloat16, "dQ after a timed-out call")
    for l in range(3):
        check(g["dK"][l], ref["dK"][l], torch.bfloat16, f"dK{l} after a timed-out call")
        check(g["dV"][l], ref["dV"][l], torch.bfloat16, f"dV{l} after a timed-out call")


@pytest.mark.parametrize("d", [128, 64])
def test_backward_wait_runs_out_in_a_later_item(mka, orc, short_limit, d):
    """160 key tiles on 148 CTAs, only the newest of them seen by a query: every CTA's first item has no tile, and the wait
    that runs out is one of a CTA's second item."""
    B, H, T, W, N = 1, 1, 300, 96, (20480, 0, 0)
    P = problem(94, B, H, T, d, N, 32, torch.bfloat16, router_std=0.3, with_dO=True)
    gate = mka.mka_router(P["X"], P["W_r"], None)
    mk = lambda flags: mka.make_shape(B, H, T, d, 32, W, q_offset=N[0] - T, flags=flags)  # noqa: E731
    shape, stalled = mk(0), mk(mka.MKA_FLAG_TEST_STALL)
    O, LSE = mka.mka_fwd(shape, P["Q"], P["K"], P["V"], gate)
    assert mka.mka_bwd_kernel_kind(shape, P["K"], P["V"]) == 1
    ws = mka.alloc_workspace(shape, N, mka.MKA_WS_BWD, "cuda")
    mka.mka_bwd(stalled, P["Q"], P["K"], P["V"], gate, O, LSE, P["dO"], ws=ws)
    assert mka.mka_device_status(ws) == MKA_ERR_TIMEOUT
    g = mka.mka_bwd(shape, P["Q"], P["K"], P["V"], gate, O, LSE, P["dO"], ws=ws)
    assert mka.mka_device_status(ws) == 0
    ref = orc.bwd(P["Q"], P["K"], P["V"], np64(gate), P["dO"], W, q_offset=N[0] - T)
    check(g["dQ"], ref["dQ"], torch.bfloat16, "dQ after a timed-out call")
    check(g["dK"][0], ref["dK"][0], torch.bfloat16, "dK after a timed-out call")
    check(g["dV"][0], ref["dV"][0], torch.bfloat16, "dV after a timed-out call")
    assert not g["dK"][0][:, :, :N[0] - T - W].any()             # the items without a tile are written, as zeros


@pytest.mark.parametrize("d", [128, 64])
def test_paged_decode_wait_runs_out_and_the_next_call_is_correct(mka, orc, short_limit, d):
    """The last tile of every CTA's share never arrives: the computing warps give up with other copies of the ring in flight."""
    B, H, Hkv, N, page = 2, 4, 2, (300, 70000, 100), 16
    P = problem(95, B, H, 1, d, N, 64, torch.bfloat16, router_std=0.3)
    gate = mka.mka_router(P["X"], P["W_r"], None).view(B, 3)
    q = P["Q"][:, :, 0].contiguous()
    pools, tabs = ([], []), []
    for l, n in enumerate(N):
        width = -(-n // page)
        tab = torch.randperm(B * width, generator=torch.Generator().manual_seed(l)).view(B, width).to(torch.int32).cuda()
        for dst, src in zip(pools, (P["K"][l][:, :Hkv], P["V"][l][:, :Hkv])):
            rows = torch.nn.functional.pad(src, (0, 0, 0, width * page - n)).view(B, Hkv, width, page, d).transpose(1, 2)
            dst.append(torch.empty(B * width, Hkv, page, d, dtype=src.dtype, device="cuda"))
            dst[-1][tab.long().flatten()] = rows.reshape(B * width, Hkv, page, d)
        tabs.append(tab)
    shape, stalled = mka.make_shape(B, H, 1, d), mka.make_shape(B, H, 1, d, flags=mka.MKA_FLAG_TEST_STALL)
    ws = torch.zeros(mka.mka_decode_paged_workspace_bytes(shape, Hkv, N), dtype=torch.uint8, device="cuda")
    t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    t0.record()
    mka.mka_decode_paged(stalled, Hkv, q, *pools, tabs, N, gate, ws=ws)
    t1.record()
    assert mka.mka_device_status(ws) == MKA_ERR_TIMEOUT
    assert t0.elapsed_time(t1) < 1000.0
    O, LSE = mka.mka_decode_paged(shape, Hkv, q, *pools, tabs, N, gate, ws=ws)
    assert mka.mka_device_status(ws) == 0
    rep = [[x[:, :Hkv].repeat_interleave(H // Hkv, 1) for x in P[k]] for k in ("K", "V")]
    Or, Lr = orc.fwd(P["Q"], *rep, np64(gate).reshape(B, 1, 3), 1, decode=True)
    check(O, Or[:, :, 0], torch.bfloat16, "paged decode after a timed-out call")
    assert np.abs(np64(LSE) - Lr[:, :, 0]).max() <= 2e-3


def test_summary_look_back_runs_out_and_the_next_call_is_correct(mka, orc, short_limit):
    B, T, D = 1, 2048, 256                                        # eight 256-row segments (or four of 512) per strip
    from mka_inputs import approx_normal
    X = approx_normal(92, 0, 0, B * T * D, 1.0, "cpu", torch.bfloat16).view(B, T, D).cuda()
    ws = mka.mka_l2_summary_workspace(X).zero_()
    assert mka.mka_l2_summary_kernel_kind(X, ws) == 1
    mka.mka_l2_summary(X, mka.MKA_SUMMARY_MEAN | mka.MKA_SUMMARY_TEST_STALL, ws=ws)
    assert mka.mka_device_status(ws) == MKA_ERR_TIMEOUT
    M2 = mka.mka_l2_summary(X, mka.MKA_SUMMARY_MEAN, ws=ws)
    assert mka.mka_device_status(ws) == 0
    ref = orc.l2_summary(np64(X))[0]
    check(M2, ref, torch.bfloat16, "summary after a timed-out call")


@pytest.mark.parametrize("d", [128, 64])
def test_a_low_limit_does_not_end_a_call_whose_pieces_are_long(mka, d):
    """Equal ranges of key tiles: a CTA works on pieces of some 280 and 240 tiles, each several times as long as the limit, while every wait
    of its copies and products is over after a tile or two.  Nothing may give up."""
    B, H, Hkv, T, q_off = 1, 24, 4, 1024, 100000
    N = (0, q_off + T, 64)
    g = torch.Generator(device="cuda").manual_seed(96)
    mk = lambda *n: torch.randn(*n, device="cuda", dtype=torch.bfloat16, generator=g)
    Q, K, V = mk(B, H, T, d), [mk(B, Hkv, n, d) for n in N], [mk(B, Hkv, n, d) for n in N]
    gate = torch.softmax(torch.randn(B, T, 3, device="cuda", generator=g), -1).contiguous()
    shape = mka.make_shape(B, H, T, d, 64, 64, q_off, kv_heads=Hkv)
    assert mka.lib.mka_fwd_scratch_bytes(ctypes.byref(shape), 0, (ctypes.c_int64 * 3)(*N)) > 0
    ws = torch.zeros(256, dtype=torch.uint8, device="cuda")
    want, want_lse = mka.mka_fwd(shape, Q, K, V, gate, ws=ws)
    assert mka.mka_device_status(ws) == 0
    old = mka.mka_set_wait_limit_us(200)
    try:
        got, lse = mka.mka_fwd(shape, Q, K, V, gate, ws=ws)
    finally:
        mka.mka_set_wait_limit_us(old)
    assert mka.mka_device_status(ws) == 0
    assert torch.equal(got, want) and torch.equal(lse, want_lse)


@pytest.mark.parametrize("case", [(1, 12, 4, 949, 128, 1750, 3804, 144), (2, 32, 32, 627, 64, 2630, 0, 7815)], ids=["d128", "d64"])
def test_forward_wait_runs_out_within_ranges(mka, short_limit, case):
    """Equal ranges of key tiles: half of the CTAs never get the last tile of their first piece, with the dealing warp at its wait, the others
    that of their second."""
    B, H, Hkv, T, d, W, q_off, n3 = case
    N = (q_off + T, q_off + T, n3)
    g = torch.Generator(device="cuda").manual_seed(97)
    mk = lambda *n: torch.randn(*n, device="cuda", dtype=torch.bfloat16, generator=g)
    Q, K, V = mk(B, H, T, d), [mk(B, Hkv, n, d) for n in N], [mk(B, Hkv, n, d) for n in N]
    gate = torch.softmax(torch.randn(B, T, 3, device="cuda", generator=g), -1).contiguous()
    shape, stalled = (mka.make_shape(B, H, T, d, 64, W, q_off, flags=f, kv_heads=Hkv) for f in (0, mka.MKA_FLAG_TEST_STALL))
    assert mka.lib.mka_fwd_scratch_bytes(ctypes.byref(stalled), 0, (ctypes.c_int64 * 3)(*N)) > 0
    ws = torch.zeros(256, dtype=torch.uint8, device="cuda")
    want, want_lse = mka.mka_fwd(shape, Q, K, V, gate, ws=ws)
    assert mka.mka_device_status(ws) == 0
    t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    t0.record()
    mka.mka_fwd(stalled, Q, K, V, gate, ws=ws)
    t1.record()
    assert mka.mka_device_status(ws) == MKA_ERR_TIMEOUT
    assert t0.elapsed_time(t1) < 1000.0
    got, lse = mka.mka_fwd(shape, Q, K, V, gate, ws=ws)
    assert mka.mka_device_status(ws) == 0
    assert torch.equal(got, want) and torch.equal(lse, want_lse)


@pytest.mark.parametrize("d", [128, 64])
def test_backward_wait_runs_out_with_dq_under_it(mka, short_limit, d):
    """Grouped heads whose key tiles walk 32 query tiles: dK and dV come first, and dQ's items run under their tail, which here is a wait that
    runs out."""
    B, H, Hkv, T, W, N = 1, 16, 4, 1000, 96, (1000, 1000, 160)
    g = torch.Generator(device="cuda").manual_seed(98)
    mk = lambda *n: torch.randn(*n, device="cuda", dtype=torch.bfloat16, generator=g)
    Q, dO, K, V = mk(B, H, T, d), mk(B, H, T, d), [mk(B, Hkv, n, d) for n in N], [mk(B, Hkv, n, d) for n in N]
    gate = torch.softmax(torch.randn(B, T, 3, device="cuda", generator=g), -1).contiguous()
    shape, stalled = (mka.make_shape(B, H, T, d, 64, W, flags=f, kv_heads=Hkv) for f in (0, mka.MKA_FLAG_TEST_STALL))
    O, LSE = mka.mka_fwd(shape, Q, K, V, gate)
    assert mka.mka_bwd_kernel_kind(shape, K, V) == 1
    ws = mka.alloc_workspace(shape, N, mka.MKA_WS_BWD, "cuda")
    want = mka.mka_bwd(shape, Q, K, V, gate, O, LSE, dO, ws=ws)
    assert mka.mka_device_status(ws) == 0
    t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    t0.record()
    mka.mka_bwd(stalled, Q, K, V, gate, O, LSE, dO, ws=ws)
    t1.record()
    assert mka.mka_device_status(ws) == MKA_ERR_TIMEOUT
    assert t0.elapsed_time(t1) < 1000.0
    got = mka.mka_bwd(shape, Q, K, V, gate, O, LSE, dO, ws=ws)
    assert mka.mka_device_status(ws) == 0
    assert torch.equal(got["dQ"], want["dQ"]) and torch.equal(got["dG"], want["dG"])
    for l in range(3): assert torch.equal(got["dK"][l], want["dK"][l]) and torch.equal(got["dV"][l], want["dV"][l])


def test_summary_hand_over_runs_out_and_the_next_call_is_correct(mka, orc, short_limit):
    """128 strips of eight tiles: one CTA to a strip, whose second group never hands its state on.  (This form leaves the scratch alone.)"""
    B, T, D = 1, 4096, 4096
    X = torch.randn(B, T, D, device="cuda", dtype=torch.bfloat16, generator=torch.Generator(device="cuda").manual_seed(99))
    ws = mka.mka_l2_summary_workspace(X).fill_(0x5a)
    assert mka.mka_l2_summary_kernel_kind(X, ws) == 1
    t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    t0.record()
    mka.mka_l2_summary(X, mka.MKA_SUMMARY_MEAN | mka.MKA_SUMMARY_TEST_STALL, ws=ws)
    t1.record()
    assert mka.mka_device_status(ws) == MKA_ERR_TIMEOUT
    assert t0.elapsed_time(t1) < 1000.0
    M2 = mka.mka_l2_summary(X, mka.MKA_SUMMARY_MEAN, ws=ws)
    assert mka.mka_device_status(ws) == 0 and bool((ws[256:] == 0x5a).all())
    check(M2, orc.l2_summary(np64(X))[0], torch.bfloat16, "summary after a timed-out call")

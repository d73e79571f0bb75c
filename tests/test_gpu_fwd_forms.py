"""How the forward deals its work to the CTAs: whole blocks, clusters, equal ranges with partial results in scratch memory; and
two heads of a group in one block.  Each against the oracle, through the C ABI."""
import ctypes

import numpy as np
import pytest
import torch

from gpu_helpers import check, err, np64, problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mka():
    import paper_2603_20586_b200 as m
    assert torch.cuda.is_available()
    return m


def _run(mka, shape, P, gate, N, scratch):
    """mka_fwd with `scratch` bytes of room for partial results, straight through the C entry point."""
    b = mka.binding
    O, LSE = torch.full_like(P["Q"], float("nan")), torch.full(P["Q"].shape[:3], float("nan"), device="cuda")
    ws = torch.full((256,), 0x55, dtype=torch.uint8, device="cuda")
    tmp = torch.full((max(scratch, 16) // 4,), float("nan"), device="cuda")
    b._check(b.lib.mka_fwd_with_scratch(ctypes.byref(shape), b._ptr(P["Q"]), b._levels(P["K"], P["V"]), b._ptr(gate), b._ptr(O), b._ptr(LSE),
                                        b._ptr(ws), 256, b._ptr(tmp) if scratch else None, scratch, b._stream(None)), "mka_fwd_with_scratch")
    assert mka.mka_device_status(ws) == 0
    return O, LSE


def _need(mka, shape, N):
    return int(mka.lib.mka_fwd_scratch_bytes(ctypes.byref(shape), 0, (ctypes.c_int64 * 3)(*N)))


# B, H, KV heads, T, d, window, q_offset, rows of the long-term level
CASES = [
    (1, 4, 2, 100, 128, 300, 2600, 200),       # one row tile: heads in pairs
    (1, 3, 1, 70, 128, 1000, 3000, 1),         # three heads: a pair and a half
    (2, 6, 2, 300, 128, 129, 900, 257),        # three row tiles, an odd group, two sequences
    (1, 7, 1, 512, 128, 4096, 1500, 130),      # seven heads, 256-row blocks
    (1, 2, 2, 257, 128, 64, 2000, 0),          # a block of one row; no long-term level
    (1, 4, 4, 200, 64, 128, 3000, 300),        # d = 64
    (1, 2, 1, 129, 64, 700, 1500, 40),
]


@pytest.mark.parametrize("case", CASES)
def test_forms_match_the_oracle(mka, orc, case):
    B, H, Hkv, T, d, W, q_off, n3 = case
    N = (q_off + T, q_off + T, n3)
    P = problem(71, B, H, T, d, N, 64, torch.bfloat16, router_std=0.3)
    P["K"], P["V"] = ([x[:, :Hkv].contiguous() for x in P[k]] for k in ("K", "V"))
    gate = mka.mka_router(P["X"], P["W_r"], None)
    shape = mka.make_shape(B, H, T, d, 64, W, q_off, kv_heads=Hkv)
    full = lambda x: np.repeat(np64(x), H // Hkv, axis=1)
    Or, Lr = orc.fwd(np64(P["Q"]), [full(k) for k in P["K"]], [full(v) for v in P["V"]], np64(gate), W, q_off)
    for scratch in sorted({0, _need(mka, shape, N)}):
        O, LSE = _run(mka, shape, P, gate, N, scratch)
        check(O, Or, torch.bfloat16, f"O, {scratch} bytes")
        assert err(LSE, Lr)[0] <= 2e-3


# sizes at which equal ranges are clearly the fastest: ragged rows, slots and windows, odd groups, pairs of heads
RANGES = [
    (1, 12, 4, 949, 128, 1750, 3804, 144),
    (2, 12, 4, 871, 128, 859, 2175, 3765),
    (1, 28, 4, 301, 128, 500, 20000, 0),
    (2, 32, 32, 627, 64, 2630, 0, 7815),
]


@pytest.mark.parametrize("case", RANGES)
def test_ranges_equal_whole_blocks(mka, case):
    """Both sum the same products in fp32, in another order of the tiles: O differs by a rounding to bf16 (2^-8 of values below 2),
    LSE by some 2^-22 of its size."""
    B, H, Hkv, T, d, W, q_off, n3 = case
    N = (q_off + T, q_off + T, n3)
    g = torch.Generator(device="cuda").manual_seed(5)
    mk = lambda *n: torch.randn(*n, device="cuda", dtype=torch.bfloat16, generator=g)
    P = {"Q": mk(B, H, T, d), "K": [mk(B, Hkv, n, d) for n in N], "V": [mk(B, Hkv, n, d) for n in N]}
    gate = torch.softmax(torch.randn(B, T, 3, device="cuda", generator=g), -1).contiguous()
    gate[:, ::5, 1] = 0.0                                             # rows without the session level
    shape = mka.make_shape(B, H, T, d, 64, W, q_off, kv_heads=Hkv)
    need = _need(mka, shape, N)
    assert need > 0
    a, la = _run(mka, shape, P, gate, N, need)
    b, lb = _run(mka, shape, P, gate, N, need - 256)                  # a little less than enough: as without scratch
    c, lc = _run(mka, shape, P, gate, N, 0)
    assert torch.equal(b, c) and torch.equal(lb, lc)
    assert (a.float() - c.float()).abs().max().item() <= 2.0 ** -7 and (la - lc).abs().max().item() <= 2e-5
    again, _ = _run(mka, shape, P, gate, N, need)
    assert torch.equal(a, again)


def test_scratch_is_asked_for_only_where_it_helps(mka):
    rows = lambda n: (ctypes.c_int64 * 3)(*n)
    few = mka.make_shape(1, 12, 124, 128, 64, 568, 36735, kv_heads=4)
    many = mka.make_shape(4, 32, 8192, 128, 64, 568)
    assert mka.lib.mka_fwd_scratch_bytes(ctypes.byref(few), 0, rows((36859, 36859, 99))) > 0
    assert mka.lib.mka_fwd_scratch_bytes(ctypes.byref(many), 0, rows((8192, 8192, 99))) == 0
    assert mka.lib.mka_fwd_scratch_bytes(ctypes.byref(few), 5, rows((36859, 36859, 99))) == 0          # 12 heads on 5: no such call
    assert mka.lib.mka_fwd_scratch_bytes(ctypes.byref(mka.make_shape(1, 12, 124, 96, 64, 568)), 0, rows((124, 124, 0))) == 0


@pytest.mark.parametrize("d", [64, 128])
def test_ranges_long_lists(mka, orc, d):
    """Many more CTAs than a merge fetches at a time share every block."""
    B, H, Hkv, T, W, q_off, n3 = 1, 4, 2, 20, 300, 60000, 77
    N = (q_off + T, q_off + T, n3)
    P = problem(73, B, H, T, d, N, 64, torch.bfloat16, router_std=0.3)
    P["K"], P["V"] = ([x[:, :Hkv].contiguous() for x in P[k]] for k in ("K", "V"))
    gate = mka.mka_router(P["X"], P["W_r"], None)
    shape = mka.make_shape(B, H, T, d, 64, W, q_off, kv_heads=Hkv)
    need = _need(mka, shape, N)
    assert need > 0
    O, LSE = _run(mka, shape, P, gate, N, need)
    again, _ = _run(mka, shape, P, gate, N, need)
    assert torch.equal(O, again)
    whole, lse_whole = _run(mka, shape, P, gate, N, 0)
    full = lambda x: np.repeat(np64(x), H // Hkv, axis=1)
    Or, Lr = orc.fwd(np64(P["Q"]), [full(k) for k in P["K"]], [full(v) for v in P["V"]], np64(gate), W, q_off)
    check(O, Or, torch.bfloat16, "O")
    assert err(LSE, Lr)[0] <= 2e-3 and (LSE - lse_whole).abs().max().item() <= 1e-4


def test_small_weights_of_a_row_are_kept(mka):
    """d = 64: the weights of keys 0..63 and of keys 64..127 of a tile are added up apart.  Four weights of 1 in the first half, 64 of 2^-24
    in the second: the sum is 4 + 2^-18 in fp32, and LSE misses it by the roundings of a logarithm and a product (1.5e-7 each at most);
    added to the ones, each of the small weights is lost and LSE is short by 9.5e-7."""
    B, H, T, d, n = 1, 2, 130, 64, 128
    Q, K, V = (torch.zeros(B, H, rows, d, device="cuda", dtype=torch.bfloat16) for rows in (T, n, n))
    Q[..., 0] = 1.0
    K[:, :, :64, 0], K[:, :, :4, 0], K[:, :, 64:, 0] = -1000.0, 0.0, -24.0      # log2 of the weights: a scale of ln 2 makes base 2
    V[..., 3] = 1.0
    gate = torch.tensor([0.0, 0.0, 1.0], device="cuda").repeat(B, T, 1).contiguous()
    shape = mka.make_shape(B, H, T, d, 64, 64, scale=float(np.log(2.0)))
    O, LSE = mka.mka_fwd(shape, Q, [None, None, K], [None, None, V], gate)
    assert (LSE.double() - np.log(4.0 + 2.0 ** -18)).abs().max().item() <= 4e-7
    assert torch.equal(O, torch.ones_like(O) * (torch.arange(d, device="cuda") == 3))


def test_a_stream_of_the_callers_gives_the_same_bits(mka):
    """The partial results of a call on a stream of its own lie in memory of that stream: other streams' allocations do not run into it."""
    B, H, Hkv, T, d, W, q_off, n3 = RANGES[0]
    N = (q_off + T, q_off + T, n3)
    g = torch.Generator(device="cuda").manual_seed(6)
    mk = lambda *n: torch.randn(*n, device="cuda", dtype=torch.bfloat16, generator=g)
    Q, K, V = mk(B, H, T, d), [mk(B, Hkv, n, d) for n in N], [mk(B, Hkv, n, d) for n in N]
    gate = torch.softmax(torch.randn(B, T, 3, device="cuda", generator=g), -1).contiguous()
    shape = mka.make_shape(B, H, T, d, 64, W, q_off, kv_heads=Hkv)
    need = _need(mka, shape, N)
    assert need > 0
    want, want_lse = mka.mka_fwd(shape, Q, K, V, gate)
    torch.cuda.synchronize()
    side = torch.cuda.Stream()

    class Handle:                                                     # anything that has a cuda_stream is a stream to the binding
        cuda_stream = side.cuda_stream

    for stream in (side, Handle()):
        outs = [(torch.empty_like(Q), torch.empty_like(want_lse), torch.zeros(256, dtype=torch.uint8, device="cuda")) for _ in range(8)]
        side.wait_stream(torch.cuda.current_stream())
        for O, LSE, ws in outs:
            mka.mka_fwd(shape, Q, K, V, gate, O=O, LSE=LSE, ws=ws, stream=stream)
            torch.full((need,), 255, dtype=torch.uint8, device="cuda")  # on the current stream, beside the call
        torch.cuda.synchronize()
        for O, LSE, ws in outs:
            assert mka.mka_device_status(ws) == 0 and torch.equal(O, want) and torch.equal(LSE, want_lse)

"""Gate gradient summed over the heads: by a kernel of its own behind dQ (40,000 queries under one key tile: dK and dV come first), and beside dK
and dV: a round of the CTAs and part of a second one (MORE), a remainder of a round, and a short level alone."""
import numpy as np
import pytest
import torch

from gpu_helpers import F32_MAX, err, np64, problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mka():
    import paper_2603_20586_b200 as m
    assert torch.cuda.is_available()
    return m


# B, H, T, d, window, rows of the three levels
TC = [(1, 3, 40000, 64, 16, (0, 0, 20)), (9, 2, 1100, 64, 64, (0, 0, 20)), (2, 5, 300, 128, 32, (300, 300, 130)), (1, 32, 1000, 128, 256, (1000, 0, 7)), (3, 2, 129, 64, 129, (129, 129, 0))]


@pytest.mark.parametrize("case", TC, ids=lambda c: f"T{c[2]}H{c[1]}d{c[3]}")
def test_tensor_core_sums_are_those_of_single_heads(mka, case):
    B, H, T, d, W, N = case
    P = problem(71, B, H, T, d, N, 64, torch.bfloat16, router_std=0.3, with_dO=True)
    gate = mka.mka_router(P["X"], P["W_r"], None)
    K, V = P["K"], P["V"]
    shape, single = (mka.make_shape(B, n, T, d, 64, W) for n in (H, 1))
    O, LSE = mka.mka_fwd(shape, P["Q"], K, V, gate)
    got = mka.mka_bwd(shape, P["Q"], K, V, gate, O, LSE, P["dO"])["dG"]
    want = torch.zeros_like(got)
    for h in range(H):
        one = lambda t: t[:, h:h + 1].contiguous()
        want += mka.mka_bwd(single, one(P["Q"]), [one(k) for k in K], [one(v) for v in V], gate, one(O), one(LSE), one(P["dO"]))["dG"]
    assert torch.equal(got, want)


@pytest.mark.parametrize("case", [(2, 3, 171, 32, 40, (171, 171, 5)), (1, 1, 700, 96, 9, (0, 0, 3)), (3, 7, 1, 64, 1, (1, 1, 40))], ids=lambda c: f"T{c[2]}H{c[1]}")
def test_cuda_core_sums_match_the_oracle(mka, orc, case):
    B, H, T, d, W, N = case
    P = problem(72, B, H, T, d, N, 32, torch.float32, router_std=0.3, with_dO=True)
    gate = mka.mka_router(P["X"], P["W_r"], None)
    shape = mka.make_shape(B, H, T, d, 32, W, dtype=mka.binding.MKA_F32)
    O, LSE = mka.mka_fwd(shape, P["Q"], P["K"], P["V"], gate)
    got = mka.mka_bwd(shape, P["Q"], P["K"], P["V"], gate, O, LSE, P["dO"])["dG"]
    rg, _ = orc.router(np64(P["X"]), np64(P["W_r"]))
    want = orc.bwd(P["Q"], P["K"], P["V"], rg, P["dO"], W)["dG"]
    # sums of up to T terms and H heads: the contract's bound grows with the largest of them
    assert err(got, want)[0] <= F32_MAX * max(1.0, np.abs(want).max())


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32], ids=["bf16", "f32"])
@pytest.mark.parametrize("over", ["gate", "LSE"])
def test_gate_gradient_written_over_an_operand(mka, dtype, over):
    B, H, T, d, W = 2, 3, 500, 64, 100
    P = problem(73, B, H, T, d, (T, T, 90), 32, dtype, router_std=0.3, with_dO=True)
    gate = mka.mka_router(P["X"], P["W_r"], None)
    shape = mka.make_shape(B, H, T, d, 32, W, dtype=mka.binding.MKA_BF16 if dtype == torch.bfloat16 else mka.binding.MKA_F32)
    O, LSE = mka.mka_fwd(shape, P["Q"], P["K"], P["V"], gate)
    apart = mka.mka_bwd(shape, P["Q"], P["K"], P["V"], gate, O, LSE, P["dO"])
    dG = gate if over == "gate" else LSE.view(-1)[:gate.numel()].view(gate.shape)
    got = mka.mka_bwd(shape, P["Q"], P["K"], P["V"], gate, O, LSE, P["dO"], dG=dG)
    assert got["dG"] is dG and torch.equal(dG, apart["dG"]) and torch.equal(got["dQ"], apart["dQ"])
    for l in range(3): assert torch.equal(got["dK"][l], apart["dK"][l]) and torch.equal(got["dV"][l], apart["dV"][l])


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32], ids=["bf16", "f32"])
@pytest.mark.parametrize("swap", [False, True], ids=["own", "values_over_keys"])
@pytest.mark.parametrize("T", [700, 3100])
def test_key_and_value_gradients_written_over_keys_and_values(mka, dtype, swap, T):
    B, H, d, W = 2, 6, 64, 100
    P = problem(74, B, H, T, d, (T, T, 90), 32, dtype, router_std=0.3, with_dO=True)
    gate = mka.mka_router(P["X"], P["W_r"], None)
    shape = mka.make_shape(B, H, T, d, 32, W, dtype=mka.binding.MKA_BF16 if dtype == torch.bfloat16 else mka.binding.MKA_F32)
    O, LSE = mka.mka_fwd(shape, P["Q"], P["K"], P["V"], gate)
    apart = mka.mka_bwd(shape, P["Q"], P["K"], P["V"], gate, O, LSE, P["dO"])
    dK, dV = (P["V"], P["K"]) if swap else (P["K"], P["V"])
    got = mka.mka_bwd(shape, P["Q"], P["K"], P["V"], gate, O, LSE, P["dO"], dK=dK, dV=dV)
    assert torch.equal(got["dQ"], apart["dQ"]) and torch.equal(got["dG"], apart["dG"])
    for l in range(3): assert torch.equal(dK[l], apart["dK"][l]) and torch.equal(dV[l], apart["dV"][l])


@pytest.mark.parametrize("case", [(2, 8, 2, 1000, 64, 100, 90), (2, 12, 2, 700, 128, 256, 200), (1, 2, 2, 5200, 64, 64, 40)], ids=["G4", "G6", "two_heads"])
@pytest.mark.parametrize("swap", [False, True], ids=["own", "values_over_keys"])
def test_both_orders_of_the_two_kernels_give_the_same_bits(mka, case, swap):
    """Sizes at which dK and dV come before dQ when they are written apart, and behind it when written over keys or values."""
    B, H, Hkv, T, d, W, n3 = case
    g = torch.Generator(device="cuda").manual_seed(75)
    mk = lambda *n: torch.randn(*n, device="cuda", dtype=torch.bfloat16, generator=g)
    N = (T, T, n3)
    Q, dO, K, V = mk(B, H, T, d), mk(B, H, T, d), [mk(B, Hkv, n, d) for n in N], [mk(B, Hkv, n, d) for n in N]
    gate = torch.softmax(torch.randn(B, T, 3, device="cuda", generator=g), -1).contiguous()
    shape = mka.make_shape(B, H, T, d, 64, W, kv_heads=Hkv)
    O, LSE = mka.mka_fwd(shape, Q, K, V, gate)
    apart = mka.mka_bwd(shape, Q, K, V, gate, O, LSE, dO)
    dK, dV = (V, K) if swap else (K, V)
    got = mka.mka_bwd(shape, Q, K, V, gate, O, LSE, dO, dK=dK, dV=dV)
    assert torch.equal(got["dQ"], apart["dQ"]) and torch.equal(got["dG"], apart["dG"])
    for l in range(3): assert torch.equal(dK[l], apart["dK"][l]) and torch.equal(dV[l], apart["dV"][l])


# walks of 20 and 23 query tiles, so dQ comes first; 313 and 218 pieces of sums (384 and 640 threads to a CTA) on 148 CTAs
MORE = [(16, 2, 2500, 128, 64, (0, 0, 20)), (16, 3, 2900, 64, 64, (0, 0, 130))]


@pytest.mark.parametrize("case", MORE, ids=lambda c: f"T{c[2]}H{c[1]}d{c[3]}")
def test_sums_of_a_second_round_are_taken(mka, case):
    B, H, T, d, W, N = case
    g = torch.Generator(device="cuda").manual_seed(76)
    mk = lambda *n: torch.randn(*n, device="cuda", dtype=torch.bfloat16, generator=g)
    Q, dO, K, V = mk(B, H, T, d), mk(B, H, T, d), [mk(B, H, n, d) for n in N], [mk(B, H, n, d) for n in N]
    gate = torch.softmax(torch.randn(B, T, 3, device="cuda", generator=g), -1).contiguous()
    shape, single = (mka.make_shape(B, n, T, d, 64, W) for n in (H, 1))
    O, LSE = mka.mka_fwd(shape, Q, K, V, gate)
    fresh = lambda: torch.full_like(gate, float("nan"))
    got = mka.mka_bwd(shape, Q, K, V, gate, O, LSE, dO, dG=fresh())["dG"]
    want = torch.zeros_like(got)
    for h in range(H):
        one = lambda t: t[:, h:h + 1].contiguous()
        want += mka.mka_bwd(single, one(Q), [one(k) for k in K], [one(v) for v in V], gate, one(O), one(LSE), one(dO), dG=fresh())["dG"]
    assert bool(torch.isfinite(got).all()) and torch.equal(got, want)

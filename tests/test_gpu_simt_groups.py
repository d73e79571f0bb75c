"""CUDA-core kernels with eight rows to a CTA (few blocks, walks of five tiles or more): rows around a block's eight, tiles around a
group's share, against the oracle."""
import numpy as np
import pytest
import torch

from gpu_helpers import F32_MAX, check, err, np64, problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mka():
    import paper_2603_20586_b200 as m
    assert torch.cuda.is_available()
    return m


CASES = [
    # B, H, T, d, window, rows of the long-term level
    (1, 4, 256, 64, 64, 128),
    (1, 1, 9, 32, 3, 300),           # one row past a block; most groups see one tile of one level
    (2, 2, 145, 96, 100, 33),
    (1, 3, 97, 64, 1, 257),
    (1, 2, 8, 96, 8, 255),
    (1, 2, 72, 32, 9, 46), (3, 1, 62, 96, 7, 28), (2, 2, 49, 64, 16, 91),        # walks of 5.5 to 7.6 tiles: groups without any
]


@pytest.mark.parametrize("case", CASES)
def test_forward_and_backward_match_the_oracle(mka, orc, case):
    B, H, T, d, W, n3 = case
    N = (T, T, n3)
    P = problem(67, B, H, T, d, N, 32, torch.float32, router_std=0.3, with_dO=True)
    gate = mka.mka_router(P["X"], P["W_r"], None)
    rg, _ = orc.router(np64(P["X"]), np64(P["W_r"]))
    shape = mka.make_shape(B, H, T, d, 32, W, dtype=mka.binding.MKA_F32)
    O, LSE = mka.mka_fwd(shape, P["Q"], P["K"], P["V"], gate)
    Or, Lr = orc.fwd(P["Q"], P["K"], P["V"], rg, W, 0)
    check(O, Or, torch.float32, "O")
    assert err(LSE, Lr)[0] <= F32_MAX
    full = mka.make_shape(B, H, T, d, 32, W, dtype=mka.binding.MKA_F32, mode=mka.binding.MKA_MODE_FULL)
    check(mka.mka_fwd(full, P["Q"], P["K"], P["V"], gate)[0], orc.fwd(P["Q"], P["K"], P["V"], rg, W, mode="full")[0], torch.float32, "O full")
    g = mka.mka_bwd(shape, P["Q"], P["K"], P["V"], gate, O, LSE, P["dO"], R=P["X"])
    ref = orc.bwd(P["Q"], P["K"], P["V"], rg, P["dO"], W)
    # gradients sum up to T terms each: the contract's bound grows with the largest of them
    for name, got, want in [("dQ", g["dQ"], ref["dQ"])] + [(f"d{k}{l}", g[f"d{k}"][l], ref[f"d{k}"][l]) for k in "KV" for l in range(3)]:
        assert err(got, want)[0] <= F32_MAX * max(1.0, np.abs(want).max()), name


def test_small_sums_of_the_groups_are_kept(mka):
    """Eight tiles of 32 slots, one to a group: a weight of 1 in the first, one of 0.4 * 2^-23 in each of the others.  Their sum is 1 + 2.8 * 2^-23;
    the nearest float and its logarithm (an ulp, 6e-8) leave LSE within 1e-7, added up one after the other in fp32 the seven are lost (3.3e-7)."""
    B, H, T, d, n = 1, 1, 16, 32, 256
    small = 0.4 * 2.0 ** -23
    Q, K, V = (torch.zeros(B, H, rows, d, device="cuda") for rows in (T, n, n))
    Q[..., 0] = 1.0
    K[..., 0] = -1000.0
    K[:, :, ::32, 0] = float(np.log(small))
    K[:, :, 0, 0] = 0.0
    gate = torch.tensor([0.0, 0.0, 1.0], device="cuda").repeat(B, T, 1).contiguous()
    shape = mka.make_shape(B, H, T, d, 32, 1, scale=1.0, dtype=mka.binding.MKA_F32)
    _, LSE = mka.mka_fwd(shape, Q, [None, None, K], [None, None, V], gate)
    assert (LSE.double() - np.log(1.0 + 7 * small)).abs().max().item() <= 1e-7

"""Weights of every size in every column of a key tile (part of a tile's weights are formed on the FMA pipe: whole blocks at both widths, all forms at
d = 64, dense and paged): scores that are exact in fp32 and run from 0 to -1000, so that weights run from 1 through the smallest normal number to 0."""
import ctypes

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mka():
    import paper_2603_20586_b200 as m
    assert torch.cuda.is_available()
    return m


def _run(mka, form, shape, Q, K, V, gate, n):
    B, H, _, d = Q.shape
    none = [None, None]
    rows = (ctypes.c_int64 * 3)(0, 0, n)
    need = int(mka.lib.mka_fwd_scratch_bytes(ctypes.byref(shape), 0, rows))
    assert (need > 0) == (form == "ranges") or form == "cluster"
    if form == "paged":
        page = 16
        pools = [x.view(B, H, n // page, page, d).transpose(1, 2).reshape(B * n // page, H, page, d).contiguous() for x in (K, V)]
        table = torch.arange(B * n // page, device="cuda", dtype=torch.int32).view(B, -1)
        return mka.mka_fwd_paged(shape, H, Q, none + [pools[0]], none + [pools[1]], none + [table], (0, 0, n), gate)
    if form == "cluster":                                                # without scratch memory few long lists go to clusters
        b = mka.binding
        O, LSE, ws = torch.empty_like(Q), torch.empty(Q.shape[:3], device="cuda"), torch.zeros(256, dtype=torch.uint8, device="cuda")
        b._check(b.lib.mka_fwd_with_scratch(ctypes.byref(shape), b._ptr(Q), b._levels(none + [K], none + [V]), b._ptr(gate), b._ptr(O), b._ptr(LSE),
                                            b._ptr(ws), 256, None, 0, b._stream(None)), "fwd")
        return O, LSE
    return mka.mka_fwd(shape, Q, none + [K], none + [V], gate)


@pytest.mark.parametrize("form,B,H,T,d,n", [
    ("whole", 2, 16, 300, 64, 256), ("whole", 2, 16, 300, 64, 131), ("whole", 2, 16, 300, 128, 256), ("whole", 2, 16, 300, 128, 300),
    ("paged", 2, 16, 300, 64, 256), ("paged", 2, 16, 300, 128, 288), ("cluster", 1, 16, 128, 64, 3072), ("ranges", 2, 32, 627, 64, 7815)])
def test_lse_and_zero_weights(mka, form, B, H, T, d, n):
    """LSE: a weight is off by 2^-22 of itself at most, a score of size x by x 2^-24 (the weights that count have x < 16), the sum of the weights, of which
    less than 300 are not lost beside the largest, and the logarithm by a few 2^-24 of LSE < 8: 2e-6 in all.  A weight of 2^-127 or less is exactly 0 (the polynomial gives
    subnormal numbers down to there, the special-function unit 0 from 2^-126 on): V holds 1e30 there, which nothing of may reach O."""
    i = torch.arange(n)
    j = (i * 97) % n                                                     # (97 shares no factor with the lengths)
    j[::128] = 0                                                         # every tile's largest weight is 1, wherever a list is cut
    K, V = torch.zeros(B, H, n, d), torch.zeros(B, H, n, d)
    K[..., 0] = -j.float().clamp(max=250.0).to(torch.bfloat16).float()
    zero = K[0, 0, :, 0] <= -127 * np.log(2.0) - 0.4                     # for every row: the queries multiply by 1 to 4
    formed = ((i % 128) // 4 % (4 if d == 64 else 3) == 0) & (i % 4 >= 2)  # columns of the polynomial
    assert bool((zero & formed).any()) and bool((zero & ~formed).any()) and bool((~zero & formed).any())
    V[..., 0], V[..., 1] = 1.0, torch.where(zero, torch.tensor(1e30), torch.tensor(0.0))
    Q = torch.zeros(B, H, T, d)
    Q[..., 0] = 1.0 + torch.arange(T).float() % 4
    gate = torch.tensor([0.0, 0.0, 1.0]).repeat(B, T, 1)
    up = lambda x: x.to(torch.bfloat16).cuda().contiguous()  # noqa: E731
    shape = mka.make_shape(B, H, T, d, 32, 1, scale=1.0)
    O, LSE = _run(mka, form, shape, up(Q), up(K), up(V), gate.cuda().contiguous(), n)
    s = Q[0, 0, :, :1].double() @ K[0, 0, :, :1].double().T
    want = torch.logsumexp(s, 1)
    assert (LSE.double().cpu() - want).abs().max().item() <= 2e-6
    o = O.float().cpu()
    assert (o[..., 0] - 1.0).abs().max().item() <= 2.0 ** -8
    assert not o[..., 1].any() and np.isfinite(o.numpy()).all()

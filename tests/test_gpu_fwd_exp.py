"""Weights of every size in every column of a key tile (whole blocks; part of a tile's weights are formed on the FMA pipe): scores that are exact in
fp32 and run from 0 to -600, so that weights run from 1 through the smallest normal number to 0."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mka():
    import paper_2603_20586_b200 as m
    assert torch.cuda.is_available()
    return m


@pytest.mark.parametrize("d,n", [(64, 256), (64, 131), (128, 256), (128, 300)])
def test_lse_and_zero_weights(mka, d, n):
    """LSE: a weight is off by 2^-22 of itself at most, a score of size x by x 2^-24 (the weights that count have x < 16), the sum of 300 terms and the
    logarithm by a few 2^-24 of LSE < 8: 2e-6 in all.  A weight below 2^-126 is 0: V holds 1e30 there, which nothing of may reach O."""
    B, H, T = 2, 16, 300
    j = (torch.arange(n) * 97) % n                                       # (97 shares no factor with the lengths)
    K, V = torch.zeros(B, H, n, d), torch.zeros(B, H, n, d)
    K[..., 0] = -(j.float() * 0.5).to(torch.bfloat16).float()
    V[..., 0], V[..., 1] = 1.0, torch.where(j >= 256, torch.tensor(1e30), torch.tensor(0.0))
    Q = torch.zeros(B, H, T, d)
    Q[..., 0] = 1.0 + torch.arange(T).float() % 4
    gate = torch.tensor([0.0, 0.0, 1.0]).repeat(B, T, 1)
    up = lambda x: x.to(torch.bfloat16).cuda().contiguous()  # noqa: E731
    shape = mka.make_shape(B, H, T, d, 32, 1, scale=1.0)
    O, LSE = mka.mka_fwd(shape, up(Q), [None, None, up(K)], [None, None, up(V)], gate.cuda().contiguous())
    s = Q[0, 0, :, :1].double() @ K[0, 0, :, :1].double().T
    want = torch.logsumexp(s, 1)
    assert (LSE.double().cpu() - want).abs().max().item() <= 2e-6
    o = O.float().cpu()
    assert (o[..., 0] - 1.0).abs().max().item() <= 2.0 ** -8
    assert not o[..., 1].any() and np.isfinite(o.numpy()).all()

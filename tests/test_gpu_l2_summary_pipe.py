"""The session summary where one CTA walks a strip with its groups of warps passing the state on: edges of its tiles (512 rows x 64
bytes or 256 x 128), more tiles than groups, carried states.  Against the oracle."""
import numpy as np
import pytest
import torch

from gpu_helpers import BF16_MAX, np64
from mka_inputs import approx_normal

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mka():
    import paper_2603_20586_b200 as m
    assert torch.cuda.is_available()
    return m


# 96 to 148 strips of 64 bytes (bf16: 32 columns, fp32: 16), or of 128 bytes where those are too many
@pytest.mark.parametrize("B,T,D,dtype", [(1, 3073, 3072, torch.bfloat16), (1, 513, 4736, torch.bfloat16), (3, 3584, 1184, torch.bfloat16),
                                         (2, 2049, 3584, torch.bfloat16), (1, 1537, 1536, torch.float32), (1, 4100, 2368, torch.float32)])
@pytest.mark.parametrize("kind,n_prev", [(0, 0), (0, 700), (1, 0), (1, 700)])
def test_pipe_matches_the_oracle(mka, orc, B, T, D, dtype, kind, n_prev):
    X = approx_normal(81, 0, 0, B * T * D, 1.0, "cpu", dtype).view(B, T, D).cuda()
    s0 = approx_normal(81, 1, 0, B * D, 1.0, "cpu", torch.float32).view(B, D).cuda()
    ws = mka.mka_l2_summary_workspace(X)
    ws.fill_(0x5a)                                                    # whatever the scratch holds on entry does not matter
    if mka.mka_l2_summary_kernel_kind(X, ws) != 1:
        pytest.skip("fp32 with many strips takes the strip form")
    state = s0.clone()
    M2 = mka.mka_l2_summary(X, kind, beta=0.9, state=state, n_prev=n_prev, ws=ws)
    assert mka.mka_device_status(ws) == 0
    ref, sref = orc.l2_summary(np64(X), kind, beta=0.9, state=np64(s0) if n_prev else None, n_prev=n_prev)
    tol = BF16_MAX if dtype == torch.bfloat16 else 1e-4
    assert np.abs(np64(M2) - ref).max() <= tol
    assert np.abs(np64(state) - sref).max() <= 1e-4 * max(1.0, np.abs(sref).max())

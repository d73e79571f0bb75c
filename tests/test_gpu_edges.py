"""GPU tests at the sizes where a dispatch rule or a tile changes over, against the CPU oracle."""
import numpy as np
import pytest
import torch

from gpu_helpers import err, np64, problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mka():
    import paper_2603_20586_b200 as m
    return m


@pytest.fixture(scope="module")
def orc():
    from oracle import mka_oracle
    return mka_oracle


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("rows,D", [(1, 4096), (295, 8), (296, 264), (297, 2056), (1183, 2048), (1184, 256), (1191, 3584)])
def test_router_rows_per_cta(mka, orc, dtype, rows, D):
    """One, two and eight rows to a CTA, with a last CTA that is not full and widths that leave threads idle."""
    X = problem(15, 1, 1, rows, 32, (1, 1, 1), D, dtype)["X"].view(rows, D)
    W = torch.randn(D, 3, device="cuda") * 0.05
    b = torch.tensor([0.1, -0.2, 0.05], device="cuda")
    ref, _ = orc.router(np64(X), np64(W), np64(b))
    gate = mka.mka_router(X, W, b)
    assert err(gate, ref)[0] <= 2e-6
    # the same rows one at a time: the row count moves the sums to another split, not to another row
    one = torch.cat([mka.mka_router(X[r:r + 1], W, b) for r in (0, rows // 2, rows - 1)])
    assert np.abs(np64(one) - ref[[0, rows // 2, rows - 1]]).max() <= 2e-6

"""Router: the splits of rows and columns over CTAs at the edges of their ranges."""
import pytest
import torch

pytestmark = pytest.mark.gpu


# edges of the rounds of resident CTAs (bf16 / fp32): four rows by four columns end their first at 2368 of 1024 columns (both), 1776 / 1184 of 1536, 1184 of 2056, fp32
# rows of 2568 their third at 3552; eight rows in place of four by eight columns around them; 186 rows at 1024 to 2048 columns; short rows; a row to the last CTA
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("rows,D", [(185, 1032), (186, 1032), (186, 2048), (1183, 256), (1184, 256), (2368, 1024), (2369, 1024), (4097, 1000), (1776, 1536), (1777, 1536),
                                    (1185, 2056), (2368, 2568), (2369, 2568), (3553, 2568), (1191, 4104), (2001, 5128), (4735, 2040)])
def test_router_rounds(dtype, rows, D):
    test_router_splits(dtype, rows, D)


# two rows a CTA end at 591, four of 512 threads at 1183, four of 256 threads at 4735, 5919, 8287 or 9471 by the width; widths below, at and past one pass (2048 columns)
# and such that the last pass has threads and whole warps without a column
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("rows,D", [(2, 2056), (296, 4096), (591, 3592), (592, 8), (593, 2056), (1183, 4104), (1185, 2040), (4735, 520), (4737, 264), (5919, 776), (5921, 776), (8287, 1032), (8289, 1032), (9471, 2056), (9473, 2056)])
def test_router_splits(dtype, rows, D):
    import paper_2603_20586_b200 as mka
    g = torch.Generator(device="cuda").manual_seed(rows + D)
    R = torch.randn(rows, D, device="cuda", generator=g).to(dtype)
    W = torch.randn(D, 3, device="cuda", generator=g) / D ** 0.5
    b = torch.randn(3, device="cuda", generator=g) * 0.1
    ref = torch.softmax(R.double() @ W.double() + b.double(), -1)
    # A logit is a sum of D products of standard deviation D^-1/2, far below 6: a lane adds up D / 32 of them at most, what follows (lanes, warps, bias) is
    # less than 40 sums, each rounded by 2^-24 of 6 at most; a gate moves by half of that at most, and softmax itself rounds a few times.
    bound = (D / 32 + 40) * 6 * 2.0 ** -24 / 2 + 4 * 2.0 ** -24
    gate = mka.mka_router(R, W, b)
    assert float((gate.double() - ref).abs().max()) <= bound
    assert torch.equal(gate, mka.mka_router(R, W, b))

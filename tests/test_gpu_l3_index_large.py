"""Codes of a pool large enough for the index form with sixteen loading warps: those of its slices, each small enough for the other
forms, bit for bit (sums and projections add up in one fixed order), and those of the oracle for the pages at both ends."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mka():
    import paper_2603_20586_b200 as m
    assert torch.cuda.is_available()
    return m


# (pages, KV heads, rows of a page, d, bits): 82 .. 205 MB of keys; the last batch of 64 (page, head) pairs is full, nearly empty, ragged
CASES = [(8960, 3, 24, 64, 64), (5043, 4, 32, 128, 256), (20001, 2, 16, 128, 128), (8007, 5, 16, 64, 64), (12505, 4, 16, 128, 32),
         (1367, 3, 160, 64, 256)]


@pytest.mark.parametrize("pages,H_kv,rows,d,bits", CASES, ids=lambda v: str(v))
@pytest.mark.parametrize("strided", [False, True], ids=["dense", "rows_outermost"])
def test_codes_of_a_large_pool_are_those_of_its_slices(mka, orc, pages, H_kv, rows, d, bits, strided):
    assert pages * H_kv * rows * d * 2 >= (200e6 if bits == 32 else 80e6)
    g = torch.Generator(device="cuda").manual_seed(pages + bits)
    shape = (pages, rows, H_kv, d) if strided else (pages, H_kv, rows, d)
    pool = torch.randn(shape, generator=g, device="cuda", dtype=torch.bfloat16)
    if strided: pool = pool.permute(0, 2, 1, 3)
    proj = torch.randn(bits, d, generator=g, device="cuda")
    codes = mka.mka_l3_index(pool, proj)
    parts = [mka.mka_l3_index(p, proj) for p in pool.split(max(1, int(10e6) // (H_kv * rows * d * 2)))]
    assert torch.equal(codes, torch.cat(parts))
    for end in (slice(0, 3), slice(pages - 3, pages)):
        want = orc.l3_index(pool[end].float().cpu().numpy(), proj.cpu().numpy())
        assert np.array_equal(codes[end].cpu().numpy().view(np.uint32), want)


# (pages, KV heads, rows of a page, d, bits): just past the lines from which that form is taken, 15 and 30 MB, with the widest codes for their pages
MIDDLE = [(1018, 1, 230, 64, 64), (1221, 4, 24, 64, 128), (1303, 3, 30, 64, 64), (917, 4, 16, 128, 128), (1222, 4, 24, 128, 256), (1833, 4, 32, 64, 256)]


@pytest.mark.parametrize("pages,H_kv,rows,d,bits", MIDDLE, ids=lambda v: str(v))
def test_codes_of_a_middle_pool_are_those_of_its_slices(mka, orc, pages, H_kv, rows, d, bits):
    assert (30e6 if bits == 256 else 15e6) <= pages * H_kv * rows * d * 2 <= 32e6
    g = torch.Generator(device="cuda").manual_seed(pages + bits)
    pool = torch.randn(pages, H_kv, rows, d, generator=g, device="cuda", dtype=torch.bfloat16)
    proj = torch.randn(bits, d, generator=g, device="cuda")
    codes = mka.mka_l3_index(pool, proj)
    assert torch.equal(codes, torch.cat([mka.mka_l3_index(p, proj) for p in pool.split(max(1, int(10e6) // (H_kv * rows * d * 2)))]))
    for end in (slice(0, 3), slice(pages - 3, pages)):
        want = orc.l3_index(pool[end].float().cpu().numpy(), proj.cpu().numpy())
        assert np.array_equal(codes[end].cpu().numpy().view(np.uint32), want)

"""Paged decode where one warp finds a CTA's share (32 sequences at most) and beyond, with sequences that have no row, closed levels, shares that
end inside a list, and lists of more partials than are asked for at once; against 64-bit arithmetic."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mka():
    import paper_2603_20586_b200 as m
    assert torch.cuda.is_available()
    return m


@pytest.mark.parametrize("B,H,Hkv,d,n2", [
    (1, 8, 1, 128, 19100),        # 299 tiles, two to a share: 150 partials of one list
    (1, 5, 1, 64, 64 * 296 * 2),  # even shares
    (2, 8, 2, 64, 5000), (3, 16, 1, 128, 130), (31, 4, 2, 128, 700), (32, 8, 2, 64, 333), (33, 8, 2, 64, 333), (40, 4, 4, 128, 65),
    (8, 16, 8, 128, 700), (2, 8, 4, 64, 900), (1, 8, 4, 64, 900)])     # few partials in four groups (d = 128), 38 in one and 75 in four (d = 64)
def test_matches_64_bits(mka, B, H, Hkv, d, n2):
    """O is a bf16 rounding (2^-9 of |O| <= 4) and weights rounded to bf16 for the product away from the exact value; LSE only fp32 sums."""
    g = torch.Generator(device="cuda").manual_seed(B * 100 + d)
    page, N = 16, (100, n2, 40)
    rows = [torch.randint(1, n + 1, (B,), device="cuda", generator=g, dtype=torch.int32) for n in N]
    rows[1][0] = n2
    if B > 2:
        for r in rows:
            r[1] = 0                                                    # a sequence without a row
    gate = torch.softmax(torch.randn(B, 3, device="cuda", generator=g), -1)
    gate[B - 1] = torch.tensor([0.0, 1.0, 0.0], device="cuda")
    pools, tabs = ([], []), []
    for n in N:
        width = -(-n // page)
        tabs.append(torch.randperm(B * width, device="cuda", generator=g).to(torch.int32).view(B, width).contiguous())
        for p in pools:
            p.append(torch.randn(B * width, Hkv, page, d, device="cuda", dtype=torch.bfloat16, generator=g))
    q = torch.randn(B, H, d, device="cuda", dtype=torch.bfloat16, generator=g)
    shape = mka.make_shape(B, H, 1, d)
    ws = torch.full((mka.mka_decode_paged_workspace_bytes(shape, Hkv, N),), 0xff, dtype=torch.uint8, device="cuda")   # NaN where nothing is written
    O, LSE = mka.mka_decode_paged(shape, Hkv, q, *pools, tabs, N, gate, rows=rows, ws=ws)
    assert mka.mka_device_status(ws) == 0
    again, _ = mka.mka_decode_paged(shape, Hkv, q, *pools, tabs, N, gate, rows=rows, ws=ws)
    assert torch.equal(O, again)
    for b in range(B):
        x, v = [], []
        for l in range(3):
            m = int(rows[l][b])
            if m == 0 or gate[b, l] == 0:
                continue
            k64, v64 = (p[l][tabs[l][b].long()].transpose(0, 1).reshape(Hkv, -1, d)[:, :m].double() for p in pools)
            x.append(q[b].double().view(Hkv, -1, d) @ k64.transpose(1, 2) * d ** -0.5 + torch.log(gate[b, l].double()))
            v.append(v64)
        if not x:
            assert not O[b].any() and torch.isinf(LSE[b]).all()
            continue
        x, v = torch.cat(x, 2), torch.cat(v, 1)
        assert (LSE[b].double() - torch.logsumexp(x, 2).view(-1)).abs().max().item() <= 1e-5
        want = (torch.softmax(x, 2) @ v).view(H, d)
        assert (O[b].double() - want).abs().max().item() <= 2e-2 and (O[b].double() - want).abs().mean().item() <= 2e-3


@pytest.mark.parametrize("paged,B,H,Hkv,d", [(True, 1, 8, 1, 128), (True, 3, 6, 2, 64), (True, 33, 4, 2, 64), (False, 2, 8, 2, 128), (False, 1, 28, 4, 64)])
def test_workspace_at_any_multiple_of_four_bytes(mka, paged, B, H, Hkv, d):
    """Partial results and the status word are written and read 4 bytes at a time: a slice of a caller's arena will do, and gives the same bits."""
    g = torch.Generator(device="cuda").manual_seed(B + d)
    mk = lambda *n: torch.randn(*n, device="cuda", dtype=torch.bfloat16, generator=g)
    N, page = (160, 2096, 48), 16
    q, gate = mk(B, H, d), torch.softmax(torch.randn(B, 3, device="cuda", generator=g), -1)
    if paged:
        shape = mka.make_shape(B, H, 1, d)
        pools = [[mk(B * n // page, Hkv, page, d) for n in N] for _ in range(2)]
        tabs = [torch.arange(B * n // page, device="cuda", dtype=torch.int32).view(B, n // page) for n in N]
        nbytes = mka.mka_decode_paged_workspace_bytes(shape, Hkv, N)
        run = lambda ws: mka.mka_decode_paged(shape, Hkv, q, *pools, tabs, N, gate, ws=ws)
    else:
        shape = mka.make_shape(B, H, 1, d, kv_heads=Hkv)
        K, V = ([mk(B, Hkv, n, d) for n in N] for _ in range(2))
        nbytes = mka.mka_workspace_bytes(shape, N, mka.MKA_WS_DECODE)
        run = lambda ws: mka.mka_decode(shape, q, K, V, gate, ws=ws)
    arena = torch.full((nbytes + 16,), 0xff, dtype=torch.uint8, device="cuda")
    want = run(arena[:nbytes])
    for off in (4, 8, 12):
        arena.fill_(0xff)
        ws = arena[off:off + nbytes]
        O, LSE = run(ws)
        assert mka.mka_device_status(ws) == 0
        assert torch.equal(O, want[0]) and torch.equal(LSE, want[1])
        assert bool((arena[:off] == 0xff).all()) and bool((arena[off + nbytes:] == 0xff).all())

"""A key with a NaN or an infinity, at every column of a key tile: each row that sees a score of NaN or +inf ends as O = 0 with LSE = -inf, whatever
the form of the call and however that column's weight is formed; rows that do not see it, and rows whose score is -inf, are as they are without."""
import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mka():
    import paper_2603_20586_b200 as m
    assert torch.cuda.is_available()
    return m


# form, B, H, KV heads, T, d, rows of the session level, tile of the key (negative: from the end; the last tile is masked for some rows)
CASES = [
    ("whole", 8, 16, 16, 128, 64, 256, 0), ("whole", 8, 16, 16, 128, 64, 256, -1), ("whole", 8, 16, 16, 128, 64, 384, 1),
    ("whole", 8, 16, 16, 128, 128, 256, 0), ("whole", 8, 16, 16, 128, 128, 256, -1), ("whole", 8, 16, 16, 300, 128, 384, 1),
    ("paged", 8, 16, 16, 128, 64, 256, -1), ("paged", 8, 16, 16, 128, 128, 256, -1), ("paged", 4, 32, 32, 128, 128, 384, 1),
    ("cluster", 1, 16, 16, 128, 64, 3072, 11), ("cluster", 1, 16, 16, 128, 64, 3072, -1),
    ("cluster", 1, 16, 16, 128, 128, 3072, 11), ("cluster", 1, 16, 16, 128, 128, 3072, -1),
    ("ranges", 2, 32, 32, 627, 64, 7815, 30), ("ranges", 1, 56, 14, 256, 128, 12800, 50),
    ("ranges of one tile", 1, 56, 14, 256, 128, 12800, 0), ("paged", 2, 32, 32, 640, 64, 7808, 30), ("paged", 1, 56, 14, 256, 128, 12800, 50),
]


@pytest.mark.parametrize("value", [float("nan"), float("inf")], ids=["nan", "inf"])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "-".join(map(str, c)))
def test_rows_that_see_the_key(mka, case, value):
    form, B, H, Hkv, T, d, n, tile = case
    g = torch.Generator(device="cuda").manual_seed(n + d)
    mk = lambda *size: torch.randn(*size, device="cuda", dtype=torch.bfloat16, generator=g)
    Q, K0, V = mk(B, H, T, d), mk(B, Hkv, n, d), mk(B, Hkv, n, d)
    Q[..., 0] = torch.where(Q[..., 0] > 0, 1.0, -1.0)                       # the sign of the scores of an infinite key
    gate = torch.softmax(torch.randn(B, T, 3, device="cuda", generator=g), -1).contiguous()
    q_off = n - T
    shape = mka.make_shape(B, H, T, d, 32, 64, q_off, kv_heads=Hkv)
    need = int(mka.lib.mka_fwd_scratch_bytes(ctypes.byref(shape), 0, (ctypes.c_int64 * 3)(0, n, 0)))
    assert need > 0 or not form.startswith("ranges")
    page = 16

    def run(K):
        if form == "paged":
            pages = lambda x: x.view(B, Hkv, n // page, page, d).transpose(1, 2).reshape(B * n // page, Hkv, page, d)
            table = torch.arange(B * n // page, device="cuda", dtype=torch.int32).view(B, -1)
            return mka.mka_fwd_paged(mka.make_shape(B, H, T, d, 32, 64, q_off), Hkv, Q, [None, pages(K), None], [None, pages(V), None],
                                     [None, table, None], (0, n, 0), gate)
        if form.startswith("ranges"):
            return mka.mka_fwd(shape, Q, [None, K, None], [None, V, None], gate)
        b = mka.binding                                                    # without scratch: few long lists go to clusters
        O, LSE = torch.empty_like(Q), torch.empty(B, H, T, device="cuda")
        ws = torch.zeros(256, dtype=torch.uint8, device="cuda")
        b._check(b.lib.mka_fwd_with_scratch(ctypes.byref(shape), b._ptr(Q), b._levels([None, K, None], [None, V, None]), b._ptr(gate), b._ptr(O),
                                            b._ptr(LSE), b._ptr(ws), 256, None, 0, b._stream(None)), "fwd")
        return O, LSE

    first = (tile if tile >= 0 else -(-n // 128) + tile) * 128
    columns = [c for c in range(128) if first + c < n]
    lines, t = B * Hkv, torch.arange(T, device="cuda")
    for at in range(0, len(columns), lines):
        here = columns[at:at + lines]
        K, big = K0.clone(), K0.clone()
        hit = torch.zeros(B, Hkv, T, dtype=torch.bool, device="cuda")
        for i, c in enumerate(here):
            b, h = i // Hkv, i % Hkv
            K[b, h, first + c, 0] = value
            big[b, h, first + c, 0] = 3e38                                  # the finite key whose weight is 0 where the infinite one's is
            hit[b, h] = t + q_off >= first + c
        hit = hit.repeat_interleave(H // Hkv, 1)
        if value == float("inf"):
            negative = hit & (Q[..., 0] < 0)
            hit &= Q[..., 0] > 0
        O, LSE = run(K)
        assert not O[hit].any() and bool((LSE[hit] == -float("inf")).all())
        Ob, Lb = run(big if value == float("inf") else K0)
        assert torch.equal(O[~hit], Ob[~hit]) and torch.equal(LSE[~hit], Lb[~hit]) and bool(torch.isfinite(LSE[~hit]).all())
        assert bool(hit.any()) and (value != float("inf") or bool(negative.any()))

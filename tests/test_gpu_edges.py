"""GPU tests at the sizes where a dispatch rule or a tile changes over, against the CPU oracle."""
import numpy as np
import pytest
import torch

from gpu_helpers import check, err, np64, problem

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
@pytest.mark.parametrize("rows,D", [(1, 4096), (295, 8), (296, 264), (297, 2056), (1183, 2048), (1184, 256), (1191, 3584), (4735, 64), (4739, 520)])
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


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("B,H,Hkv,T,W,q_off,N", [
    (1, 2, 2, 130, 700, 1870, (2000, 2000, 300)),        # a few blocks, long lists: the widest cluster
    (1, 4, 1, 257, 129, 1000, (1257, 1257, 0)),          # a block with one row, no long-term level, window edges inside
    (1, 1, 1, 1, 1, 900, (901, 901, 1)),                 # one row; the window is its own tile
    (2, 20, 4, 300, 64, 0, (300, 300, 2100)),            # the first rows see little of a list that the long-term level fills
    (1, 3, 3, 64, 5000, 4000, (4064, 100, 17)),          # window wider than the level, short session level
])
def test_fwd_key_tiles_split_between_ctas(mka, orc, d, B, H, Hkv, T, W, q_off, N):
    """Few blocks of query rows: the key-tile list is split over a cluster and merged (also in its ragged and masked parts)."""
    P = problem(31, B, H, T, d, N, 64, torch.bfloat16, router_std=0.5)
    K, V = ([x[:, :Hkv].contiguous() for x in P[k]] for k in ("K", "V"))
    shape = mka.make_shape(B, H, T, d, 64, W, q_off, kv_heads=Hkv)
    assert mka.mka_fwd_kernel_kind(shape, K, V) == 1
    for route in (mka.binding.MKA_ROUTE_SOFT, mka.binding.MKA_ROUTE_TOP1):      # TOP1: whole levels weigh 0 for a row
        gate = mka.mka_router(P["X"], P["W_r"], None, route=route)
        ws = mka.alloc_workspace(shape, N, mka.binding.MKA_WS_FWD, "cuda")
        O, LSE = mka.mka_fwd(shape, P["Q"], K, V, gate, ws=ws)
        assert mka.mka_device_status(ws) == 0
        rep = [[x.repeat_interleave(H // Hkv, 1) for x in t] for t in (K, V)]
        Or, Lr = orc.fwd(P["Q"], rep[0], rep[1], np64(gate), W, q_off)
        check(O, Or, torch.bfloat16, "O")
        finite = np.isfinite(Lr)
        assert np.array_equal(np.isfinite(np64(LSE)), finite)
        assert np.abs(np64(LSE)[finite] - Lr[finite]).max() <= 2e-3
        again, _ = mka.mka_fwd(shape, P["Q"], K, V, gate, ws=ws)
        assert torch.equal(O, again)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("B,H,Hkv,T,W,q_off,N", [
    (4, 16, 4, 700, 64, 600, (1300, 1600, 40)),          # keys that no query sees (left of every window, past the last query): items without a tile
    (5, 8, 8, 1100, 200, 0, (1100, 1100, 300)),          # one and more tiles to an item, last tiles that are not full
])
def test_bwd_items_carried_over(mka, orc, d, B, H, Hkv, T, W, q_off, N):
    """More than two output tiles to every CTA of the dQ and the dK/dV kernel: rings, buffers and barriers go on from item to item.
    The result may not change from call to call either: a tile read before every warp has written its part would."""
    assert B * H * -(-T // 128) > 296 and B * Hkv * sum(-(-n // 128) for n in N) > 296
    P = problem(43, B, H, T, d, N, 64, torch.bfloat16, router_std=0.5, with_dO=True)
    K, V = ([x[:, :Hkv].contiguous() for x in P[k]] for k in ("K", "V"))
    shape = mka.make_shape(B, H, T, d, 64, W, q_off, kv_heads=Hkv)
    assert mka.mka_bwd_kernel_kind(shape, K, V) == 1
    gate = mka.mka_router(P["X"], P["W_r"], None)
    O, LSE = mka.mka_fwd(shape, P["Q"], K, V, gate)
    ws = mka.alloc_workspace(shape, N, mka.MKA_WS_BWD, "cuda")
    run = lambda: mka.mka_bwd(shape, P["Q"], K, V, gate, O, LSE, P["dO"], R=P["X"], ws=ws)  # noqa: E731
    g = run()
    assert mka.mka_device_status(ws) == 0
    for _ in range(20):
        again = run()
        assert torch.equal(g["dQ"], again["dQ"])
        for l in range(3):
            assert torch.equal(g["dK"][l], again["dK"][l]) and torch.equal(g["dV"][l], again["dV"][l])
    G = H // Hkv
    rep = [[x.repeat_interleave(G, 1) for x in t] for t in (K, V)]
    r = orc.bwd(P["Q"], rep[0], rep[1], np64(gate), P["dO"], W, q_off)
    check(g["dQ"], r["dQ"], torch.bfloat16, "dQ")
    for l in range(3):
        for name in ("dK", "dV"):
            want = r[name][l].reshape(B, Hkv, G, N[l], d).sum(2)
            # one rounding to bf16 of a sum over the group's heads and up to T queries: half a step of the largest value, on top of the contract's bound
            mx, mean = err(g[name][l], want)
            assert mx <= 2e-2 + np.abs(want).max() / 256 and mean <= 2e-3 + np.abs(want).mean() / 256, (name, l, mx, mean)
    check(g["dG"], r["dG"], torch.bfloat16, "dG")


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("B,T,D", [(1, 1, 64), (1, 127, 264), (2, 300, 2048), (3, 1111, 1000), (1, 5000, 256), (2, 70, 100)])
def test_router_gradient_splits(mka, orc, dtype, B, T, D):
    """dW_r and db_r: row chunks without a row, batches that end inside a chunk, column blocks that are not full."""
    H, d, N = 1, 64, (T, T, 40)
    P = problem(17, B, H, T, d, N, D, dtype, router_std=0.3, with_dO=True)
    gate = mka.mka_router(P["X"], P["W_r"], None)
    shape = mka.make_shape(B, H, T, d, D, 32, dtype=mka.binding.MKA_BF16 if dtype == torch.bfloat16 else mka.binding.MKA_F32)
    O, LSE = mka.mka_fwd(shape, P["Q"], P["K"], P["V"], gate)
    g = mka.mka_bwd(shape, P["Q"], P["K"], P["V"], gate, O, LSE, P["dO"], R=P["X"])
    dG = np64(g["dG"])
    dW, db = orc.router_bwd(np64(P["X"]), dG)
    # fp32 sums of B T products: the bound is their number times the unit roundoff times the sum of magnitudes
    mag = np.abs(np64(P["X"]).reshape(-1, D)).T @ np.abs(dG.reshape(-1, 3))
    assert (np.abs(np64(g["dW_r"]) - dW) <= (B * T + 130) * 6e-8 * mag + 1e-30).all()
    assert (np.abs(np64(g["db_r"]) - db) <= 6e-8 * np.abs(db) + 1e-15 * np.abs(dG).sum() * B * T).all()


def test_bwd_workspace_alignment(mka, orc):
    """fp32 takes a workspace at any word; the tensor-core kernels read their statistics 16 bytes at a time and refuse what allows none."""
    B, H, T, d, N, D = 1, 2, 130, 64, (130, 130, 40), 72
    for dtype in (torch.float32, torch.bfloat16):
        P = problem(18, B, H, T, d, N, D, dtype, router_std=0.3, with_dO=True)
        gate = mka.mka_router(P["X"], P["W_r"], None)
        shape = mka.make_shape(B, H, T, d, D, 32, dtype=mka.binding.MKA_BF16 if dtype == torch.bfloat16 else mka.binding.MKA_F32)
        O, LSE = mka.mka_fwd(shape, P["Q"], P["K"], P["V"], gate)
        ws = mka.alloc_workspace(shape, N, mka.MKA_WS_BWD, "cuda")
        off = torch.zeros(ws.numel() + 4, dtype=torch.uint8, device="cuda")[4:]
        run = lambda w: mka.mka_bwd(shape, P["Q"], P["K"], P["V"], gate, O, LSE, P["dO"], R=P["X"], ws=w)  # noqa: E731
        want = run(ws)
        if dtype == torch.bfloat16:
            with pytest.raises(RuntimeError, match="align"):
                run(off)
            continue
        got = run(off)
        for k in ("dQ", "dG", "dW_r"):
            assert torch.equal(got[k], want[k])
        # one CTA's sum of dG in place of the chunks' sums, both in 64 bits: one rounding apart at most
        assert err(got["db_r"], np64(want["db_r"]))[0] <= 1.2e-7 * np.abs(np64(want["db_r"])).max()


@pytest.mark.parametrize("d,dtype,shift", [(32, torch.float32, 0), (64, torch.float32, 1), (96, torch.float32, 0), (128, torch.float32, 3),
                                           (96, torch.bfloat16, 0), (32, torch.bfloat16, 0)])
@pytest.mark.parametrize("T,W,q_off,N", [(1, 1, 0, (1, 1, 0)), (17, 5, 300, (317, 317, 33)), (130, 64, 0, (130, 100, 31))])
def test_cuda_core_tiles(mka, orc, d, dtype, shift, T, W, q_off, N):
    """CUDA-core kernels: rows and tiles that are not full, groups without a tile, float tensors that allow no 16-byte load."""
    B, H = 2, 3
    P = problem(23, B, H, T, d, N, 64, dtype, router_std=0.5, with_dO=True)

    def moved(x):                       # the same values at an address `shift` floats off
        if not shift:
            return x
        buf = torch.empty(x.numel() + shift, dtype=x.dtype, device=x.device)
        out = buf[shift:].view(x.shape)
        return out.copy_(x)

    Q, dO, K, V = moved(P["Q"]), moved(P["dO"]), [moved(k) for k in P["K"]], [moved(v) for v in P["V"]]
    gate = mka.mka_router(P["X"], P["W_r"], None)
    mk = lambda mode: mka.make_shape(B, H, T, d, 64, W, q_off, dtype=mka.binding.MKA_BF16 if dtype == torch.bfloat16 else mka.binding.MKA_F32,  # noqa: E731
                                     mode=mode)
    shape, full = mk(mka.binding.MKA_MODE_FAST), mk(mka.binding.MKA_MODE_FULL)
    assert mka.mka_fwd_kernel_kind(shape, K, V) == 0
    O, LSE = mka.mka_fwd(shape, Q, K, V, gate)
    g64 = np64(gate)
    Or, Lr = orc.fwd(P["Q"], P["K"], P["V"], g64, W, q_off)
    check(O, Or, dtype, "O")
    assert err(LSE, Lr)[0] <= 1e-4
    check(mka.mka_fwd(full, Q, K, V, gate)[0], orc.fwd(P["Q"], P["K"], P["V"], g64, W, q_off, mode="full")[0], dtype, "O of the per-level form")
    g = mka.mka_bwd(shape, Q, K, V, gate, O, LSE, dO, R=P["X"])
    r = orc.bwd(P["Q"], P["K"], P["V"], g64, P["dO"], W, q_off)
    check(g["dQ"], r["dQ"], dtype, "dQ")
    for l in range(3):
        if N[l]:
            check(g["dK"][l], r["dK"][l], dtype, f"dK{l}")
            check(g["dV"][l], r["dV"][l], dtype, f"dV{l}")
    check(g["dG"], r["dG"], dtype, "dG")


@pytest.mark.parametrize("d,dtype", [(32, torch.float32), (64, torch.float32), (96, torch.float32), (128, torch.float32), (96, torch.bfloat16)])
@pytest.mark.parametrize("B,H,T,W,N", [
    (1, 40, 97, 9, (97, 0, 33)),           # many short walks: one group of warps to a CTA, 32 rows, the last block with one
    (2, 20, 250, 40, (250, 250, 5)),       # and a long-term level whose keys walk every query beside a short window's
])
def test_cuda_core_many_blocks(mka, orc, d, dtype, B, H, T, W, N):
    P = problem(29, B, H, T, d, N, 64, dtype, router_std=0.5, with_dO=True)
    gate = mka.mka_router(P["X"], P["W_r"], None)
    mk = lambda mode: mka.make_shape(B, H, T, d, 64, W, dtype=mka.binding.MKA_BF16 if dtype == torch.bfloat16 else mka.binding.MKA_F32, mode=mode)  # noqa: E731
    shape, full = mk(mka.binding.MKA_MODE_FAST), mk(mka.binding.MKA_MODE_FULL)
    O, LSE = mka.mka_fwd(shape, P["Q"], P["K"], P["V"], gate)
    g64 = np64(gate)
    check(O, orc.fwd(P["Q"], P["K"], P["V"], g64, W)[0], dtype, "O")
    check(mka.mka_fwd(full, P["Q"], P["K"], P["V"], gate)[0], orc.fwd(P["Q"], P["K"], P["V"], g64, W, mode="full")[0], dtype, "O of the per-level form")
    g = mka.mka_bwd(shape, P["Q"], P["K"], P["V"], gate, O, LSE, P["dO"])
    r = orc.bwd(P["Q"], P["K"], P["V"], g64, P["dO"], W)
    check(g["dQ"], r["dQ"], dtype, "dQ")
    for l in range(3):
        if N[l]:
            check(g["dK"][l], r["dK"][l], dtype, f"dK{l}")
            check(g["dV"][l], r["dV"][l], dtype, f"dV{l}")
    # dG sums over 40 (20) heads, each within the contract's bound of a single head's sum
    assert err(g["dG"], r["dG"])[0] <= (2e-2 if dtype == torch.bfloat16 else 1e-4) * H / 4


@pytest.mark.parametrize("d,bits", [(64, 32), (64, 64), (128, 64), (128, 128), (128, 256)])
@pytest.mark.parametrize("pages,H_kv,page", [(1, 1, 16), (21, 3, 8), (300, 4, 5), (1201, 4, 24), (1184, 4, 16), (1185, 4, 16), (1185, 4, 32), (20001, 2, 3)])
def test_recall_codes_batches(mka, orc, d, bits, pages, H_kv, page):
    """Recall codes: a batch with one pair, a last batch that is not full, pages of no whole number of eight rows, several batches a CTA,
    both forms of the kernel on either side of every line between them."""
    g = torch.Generator().manual_seed(3)
    pool = torch.randn(pages, H_kv, page, d, generator=g).bfloat16().cuda()
    proj = torch.randn(bits, d, generator=g).cuda()
    codes = mka.mka_l3_index(pool, proj)
    assert np.array_equal(codes.cpu().numpy().view(np.uint32), orc.l3_index(pool.float().cpu().numpy(), proj.cpu().numpy()))


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("B,H,N", [
    (1, 1, (1, 1, 0)),                 # eight CTAs, two rows
    (1, 3, (17, 300, 31)),             # slabs that are not full, levels that end inside a round
    (1, 3, (100, 16500, 200)),         # clusters of eight with about 2100 rows a CTA: the split form at d = 128
    (1, 3, (100, 40000, 200)),         # the split form at both widths
    (2, 176, (300, 900, 40)),          # more CTAs than fit, a short last round: one kernel at d = 64, two at d = 128
    (3, 40, (600, 40, 33)),            # clusters of two
    (2, 150, (130, 0, 5)),             # one CTA a pair, more CTAs than fit at once
])
def test_decode_one_kernel_or_two(mka, orc, d, B, H, N):
    P = problem(37, B, H, 1, d, N, 64, torch.bfloat16, router_std=0.5)
    q = P["Q"][:, :, 0].contiguous()
    shape = mka.make_shape(B, H, 1, d, 64)
    for route in (mka.binding.MKA_ROUTE_SOFT, mka.binding.MKA_ROUTE_TOP1):      # TOP1: levels that are not read
        gate = mka.mka_router(P["X"], P["W_r"], None, route=route).view(B, 3)
        ws = torch.full((mka.mka_workspace_bytes(shape, N, mka.binding.MKA_WS_DECODE),), 255, dtype=torch.uint8, device="cuda")
        O, LSE = mka.mka_decode(shape, q, P["K"], P["V"], gate, ws=ws)
        assert mka.mka_device_status(ws) == 0
        Or, Lr = orc.fwd(P["Q"], P["K"], P["V"], np64(gate).reshape(B, 1, 3), 1, decode=True)
        check(O, Or[:, :, 0], torch.bfloat16, "O")
        finite = np.isfinite(Lr[:, :, 0])
        assert np.array_equal(np.isfinite(np64(LSE)), finite)
        assert not finite.any() or np.abs(np64(LSE)[finite] - Lr[:, :, 0][finite]).max() <= 1e-4


@pytest.mark.parametrize("bits,n,R", [(32, 1, 8), (64, 31, 64), (64, 8191, 8), (64, 8193, 16), (128, 1025, 7), (256, 2050, 64), (32, 9000, 64), (128, 9001, 8), (256, 40000, 8)])
def test_recall_lists(mka, orc, bits, n, R):
    """Recall lists: fewer chunks than asked for, banks around a thread's chunks, few code bits (long runs of ties), a sequence with no bank."""
    B, H, H_kv, d = 3, 6, 2, 64
    g = torch.Generator().manual_seed(bits + n)
    q = torch.randn(B, H, d, generator=g).bfloat16().cuda()
    proj = torch.randn(bits, d, generator=g).cuda()
    pages = n + 5
    codes = torch.randint(-2**31, 2**31, (pages, H_kv, bits // 32), generator=g, dtype=torch.int64).to(torch.int32).cuda()
    bank = torch.stack([torch.randperm(pages, generator=g)[:n] for _ in range(B)]).to(torch.int32).cuda()
    lens = torch.tensor([n, max(1, n // 3), 0], dtype=torch.int32).cuda()
    off = lambda x: torch.cat([x.new_zeros(1), x.flatten()])[1:].view(x.shape)                  # noqa: E731  the same values at an address that allows no vector load
    for pj, cd in ((proj, codes), (off(proj), codes), (proj, off(codes))):
        table, n_sel, rows = mka.mka_l3_retrieve(q, H_kv, pj, cd, bank, lens, R, 16)
        words = codes.cpu().numpy().view(np.uint32)
        for b in range(B):
            m = int(lens[b])
            k = min(R, m)
            assert int(n_sel[b]) == k and int(rows[b]) == 16 * k
            for h in range(H_kv):
                qsum = orc.sum_rows_f32(q[b, h * 3:(h + 1) * 3].float().cpu().numpy())
                qc = orc.srp_code(qsum, proj.cpu().numpy())
                own = bank[b, :m].cpu().numpy()
                agree = bits - np.array([sum(bin(int(a ^ c)).count("1") for a, c in zip(words[pg, h], qc)) for pg in own], dtype=np.int64)
                best = sorted(sorted(range(m), key=lambda i: (-agree[i], i))[:k])
                want = np.zeros(R, dtype=np.int64)
                want[:k] = own[best]
                assert np.array_equal(table[b, h].cpu().numpy(), want)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("B,H,H_kv,N,page", [
    (1, 16, 1, (64, 1, 0), 8),             # two tiles: one share
    (37, 4, 2, (40, 130, 3), 16),          # shares that end inside lists and reach over several sequences
    (3, 14, 2, (300, 9000, 70), 64),       # lists of dozens of shares
    (150, 4, 2, (70, 129, 200), 16),       # shares of nine tiles, every third one ragged: stages refilled behind rows that were cleared
    (513, 2, 1, (20, 33, 0), 16),          # shares found through blocks of two sequences
    (2500, 2, 2, (9, 70, 0), 16),          # of eight
    (20000, 1, 1, (1, 3, 0), 8),           # and of 64, with sequences without a row among them
])
def test_decode_paged_shares(mka, orc, d, B, H, H_kv, N, page):
    """Paged decode against the dense oracle: mixed lengths, sequences without a row, levels that a gate closes."""
    P = problem(41, B, H, 1, d, N, 64, torch.bfloat16, router_std=0.5)
    q = P["Q"][:, :, 0].contiguous()
    gate = mka.mka_router(P["X"], P["W_r"], None).view(B, 3).clone()
    gate[B // 2, 1] = 0.0
    g = torch.Generator().manual_seed(5)
    rows = [torch.randint(0, n + 1, (B,), generator=g, dtype=torch.int32) for n in N]
    for r, n in zip(rows, N):
        r[0] = n
    if B > 2:
        for r in rows:
            r[B - 1] = 0
    K, V = ([x[:, :H_kv].contiguous() for x in P[k]] for k in ("K", "V"))
    pk, pv, tabs = [], [], []
    for l, n in enumerate(N):
        width = max(1, -(-n // page))
        tab = torch.randperm(B * width + 2, generator=g)[:B * width].view(B, width).to(torch.int32)
        a, b = (torch.full((B * width + 2, H_kv, page, d), float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(2))
        for s in range(B):
            for j in range(-(-int(rows[l][s]) // page)):
                m = min(page, int(rows[l][s]) - j * page)
                a[tab[s, j], :, :m] = K[l][s, :, j * page:j * page + m]
                b[tab[s, j], :, :m] = V[l][s, :, j * page:j * page + m]
        pk.append(a), pv.append(b), tabs.append(tab.cuda())
    shape = mka.make_shape(B, H, 1, d, 64)
    ws = torch.full((mka.mka_decode_paged_workspace_bytes(shape, H_kv, N),), 255, dtype=torch.uint8, device="cuda")
    O, LSE = mka.mka_decode_paged(shape, H_kv, q, pk, pv, tabs, N, gate, rows=[r.cuda() for r in rows], ws=ws)
    assert mka.mka_device_status(ws) == 0
    for _ in range(30):                    # (a row cleared or copied too late would not come out the same every time)
        again, _ = mka.mka_decode_paged(shape, H_kv, q, pk, pv, tabs, N, gate, rows=[r.cuda() for r in rows], ws=ws)
        assert torch.equal(O, again)
    for s in sorted({0, 1 % B, B // 2, B - 2 if B > 2 else 0, B - 1}):
        ks, vs = ([x[l][s:s + 1, :, :int(rows[l][s])].repeat_interleave(H // H_kv, 1) for l in range(3)] for x in (K, V))
        Or, Lr = orc.fwd(P["Q"][s:s + 1], ks, vs, np64(gate[s:s + 1]).reshape(1, 1, 3), 1, decode=True)
        seen = np.isfinite(Lr[0, 0, 0])
        check(O[s:s + 1], Or[:, :, 0] if seen else np.zeros_like(Or[:, :, 0]), torch.bfloat16, f"O of sequence {s}")
        got = np64(LSE[s:s + 1])
        assert np.isfinite(got).all() == seen
        assert not seen or np.abs(got - Lr[:, :, 0]).max() <= 1e-4

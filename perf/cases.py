"""Timed cases of the library: what a training run, a serving engine and a memory manager have it do, through the binding.

Eight kinds of pass; sizes follow the workload configurations of ``mka_inputs`` and the tests, inputs are N(0, 1) with a
router matrix of standard deviation 0.02:

    train    router, fused forward and backward of one attention layer, bf16 (head width 64 or 128, plain or grouped heads)
    fp32     the same in fp32 plus the per-level softmax form (MKA_MODE_FULL): the small-scale reference runs
    prefill  router and forward of a whole prompt against dense levels
    chunk    one chunk of a long prompt in a serving engine: router, route-fused rows appended to the paged session cache,
             forward over paged levels with grouped heads
    decode   one token per sequence against dense caches
    serve    one token per sequence in a paged serving engine: router, append of the fused row, recall of long-term chunks,
             paged grouped-query decode over window, session and recalled chunks
    summary  causal session summary of a router input (prefix mean or EMA)
    index    recall codes of a long-term key pool

Callers keep workspaces and the serving loops keep their output buffers; a training or prefill pass lets the binding
allocate its outputs, as a call in a model does.
"""
from __future__ import annotations

import torch

import paper_2603_20586_b200.binding as mka

_DEV = "cuda"
_BF16, _F32 = torch.bfloat16, torch.float32


def listed():
    return [
        # One chat turn on one sequence with a short history: the smallest call, launches and host work count.
        dict(name="decode_one", kind="decode", B=1, H=32, Hkv=32, d=128, n1=512, n2=1000, n3=64),
        # A full decode batch with long caches (the long-context decode geometry at half its batch).
        dict(name="decode_batch", kind="decode", B=16, H=32, Hkv=32, d=128, n1=4096, n2=32768, n3=8192),
        # A serving step at 128K context: Qwen2.5-7B-like heads (28 on 4), 16-row pages, top-8 recall of 8192 chunks.
        dict(name="serve_128k", kind="serve", B=4, H=28, Hkv=4, d=128, n1=4096, n2=131072, page=16, bank=8192, R=8, bits=64),
        # The whole-prompt prefill at 32K tokens: the largest call.
        dict(name="prefill_32k", kind="prefill", B=1, H=32, Hkv=32, d=128, T=32768, W=4096, n3=8192),
        # A short prompt of odd length.
        dict(name="prefill_short", kind="prefill", B=1, H=16, Hkv=16, d=64, T=777, W=512, n3=100),
        # A 512-token chunk at 15K context of a chunked prefill.
        dict(name="chunk_15k", kind="chunk", B=1, H=28, Hkv=4, d=128, T=512, ctx=15000, W=4096, n3=1024, page=16),
        # The training-shape layer, head width 64.
        dict(name="train_d64", kind="train", B=8, H=16, Hkv=16, d=64, T=2048, W=512, n3=1024),
        # The long-sequence training layer, head width 128.
        dict(name="train_d128", kind="train", B=4, H=16, Hkv=16, d=128, T=8192, W=1024, n3=2048),
        # Fine-tuning on ragged short sequences with grouped heads.
        dict(name="train_gqa", kind="train", B=2, H=16, Hkv=4, d=128, T=1000, W=256, n3=500),
        # The small fp32 configuration, both modes and the backward.
        dict(name="fp32_step", kind="fp32", B=1, H=4, d=64, T=256, W=64, n3=128),
        # Session summary of one 32K-token sequence.
        dict(name="summary_32k", kind="summary", B=1, T=32768, D=4096, bf16=True, ema=True, carry=False),
        # Recall codes of four 128K-token banks.
        dict(name="index_bank", kind="index", pages=32769, Hkv=4, page=16, d=128, bits=64),
    ]


def _log(rng, lo, hi):
    """A whole number between lo and hi, spread over the logarithm."""
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["train", "fp32", "prefill", "chunk", "decode", "serve", "summary", "index"])
    if kind == "train":
        d = rng.choice([64, 128])
        H, Hkv = rng.choice([(16, 16), (16, 4), (8, 8), (12, 4)])
        T = _log(rng, 200, 8192)
        B = max(1, min(8, int(4 * 8192 ** 2 / T ** 2 * rng.uniform(0.1, 1.0))))
        return dict(kind=kind, B=B, H=H, Hkv=Hkv, d=d, T=T, W=_log(rng, 64, 1024), n3=_log(rng, 16, 2048))
    if kind == "fp32":
        T = _log(rng, 64, 1024)
        return dict(kind=kind, B=rng.randint(1, 2), H=rng.choice([4, 8]), d=rng.choice([32, 64, 96, 128]), T=T,
                    W=max(1, T // rng.randint(2, 8)), n3=_log(rng, 16, 512))
    if kind == "prefill":
        H, Hkv = rng.choice([(16, 16), (32, 32), (28, 4), (32, 8)])
        T = _log(rng, 256, 32768)
        return dict(kind=kind, B=1 if T > 4096 else rng.randint(1, 4), H=H, Hkv=Hkv, d=rng.choice([64, 128]), T=T,
                    W=_log(rng, 256, 4096), n3=_log(rng, 64, 8192))
    if kind == "chunk":
        H, Hkv = rng.choice([(28, 4), (32, 8), (12, 4)])
        return dict(kind=kind, B=rng.randint(1, 2), H=H, Hkv=Hkv, d=128, T=_log(rng, 64, 2048), ctx=_log(rng, 1000, 60000),
                    W=_log(rng, 512, 4096), n3=_log(rng, 64, 4096), page=rng.choice([16, 32, 64]))
    if kind == "decode":
        H, Hkv = rng.choice([(32, 32), (16, 16), (28, 4), (32, 8)])
        B = _log(rng, 1, 16)
        return dict(kind=kind, B=B, H=H, Hkv=Hkv, d=rng.choice([64, 128]), n1=_log(rng, 256, 4096), n2=_log(rng, 500, 32768),
                    n3=_log(rng, 16, 8192))
    if kind == "serve":
        H, Hkv = rng.choice([(28, 4), (32, 8), (12, 4)])
        return dict(kind=kind, B=_log(rng, 1, 8), H=H, Hkv=Hkv, d=128, n1=_log(rng, 256, 4096), n2=_log(rng, 1000, 131072),
                    page=rng.choice([16, 32]), bank=_log(rng, 64, 8192), R=rng.choice([4, 8, 16]), bits=rng.choice([64, 128]))
    if kind == "summary":
        B = rng.randint(1, 4)
        ema = rng.random() < 0.5
        return dict(kind=kind, B=B, T=_log(rng, 300, 65536 // B), D=rng.choice([1024, 2048, 3584, 4096]), bf16=rng.random() < 0.75,
                    ema=ema, carry=ema and rng.random() < 0.5)
    return dict(kind=kind, pages=_log(rng, 200, 40000), Hkv=rng.choice([2, 4, 8]), page=rng.choice([8, 16, 32]), d=rng.choice([64, 128]),
                bits=rng.choice([32, 64, 128]))


class _Rng:
    def __init__(self, seed):
        self.g = torch.Generator(device=_DEV).manual_seed(int(seed))

    def normal(self, *shape, dtype=_BF16, std=1.0):
        x = torch.randn(*shape, dtype=dtype, device=_DEV, generator=self.g)
        return x if std == 1.0 else x.mul_(std)

    def perm(self, n):
        return torch.randperm(n, device=_DEV, generator=self.g).to(torch.int32)


def _router_weights(r, D):
    return r.normal(D, 3, dtype=_F32, std=0.02), torch.zeros(3, dtype=_F32, device=_DEV)


def _pool(r, B, Hkv, n, page, d):
    """A paged level: key and value pools and the sequences' page tables (pages dealt from a shuffle, a few spare)."""
    width = -(-n // page)
    pages = B * width + 3
    k, v = r.normal(pages, Hkv, page, d), r.normal(pages, Hkv, page, d)
    return k, v, r.perm(pages)[:B * width].view(B, width).contiguous()


def _lengths(B, n):
    """Rows of every sequence of a mixed batch, n the longest."""
    frac = (1.0, 0.61, 0.33, 0.87)
    return [max(1, int(n * frac[b % 4])) for b in range(B)]


def prepare(case, seed):
    c = dict(case)
    r = _Rng(seed)
    s = {"case": c}
    kind = c["kind"]
    if kind in ("train", "fp32", "prefill"):
        dt = _F32 if kind == "fp32" else _BF16
        B, H, d, T = c["B"], c["H"], c["d"], c["T"]
        Hkv = c.get("Hkv", H)
        D = H * d
        s["X"] = r.normal(B, T, D, dtype=dt)
        s["W_r"], s["b_r"] = _router_weights(r, D)
        s["Q"] = r.normal(B, H, T, d, dtype=dt)
        n = (T, T, c["n3"])
        s["K"] = [r.normal(B, Hkv, m, d, dtype=dt) for m in n]
        s["V"] = [r.normal(B, Hkv, m, d, dtype=dt) for m in n]
        mk = lambda mode: mka.make_shape(B, H, T, d, D=D, window=c["W"], dtype=mka.MKA_F32 if kind == "fp32" else mka.MKA_BF16,  # noqa: E731
                                         mode=mode, kv_heads=Hkv)
        s["shape"] = mk(mka.MKA_MODE_FAST)
        s["ws"] = mka.alloc_workspace(s["shape"], n, mka.MKA_WS_FWD, _DEV)
        if kind != "prefill":
            s["dO"] = r.normal(B, H, T, d, dtype=dt)
            s["ws_bwd"] = mka.alloc_workspace(s["shape"], n, mka.MKA_WS_BWD, _DEV)
        if kind == "fp32":
            s["shape_full"] = mk(mka.MKA_MODE_FULL)
    elif kind == "chunk":
        B, H, Hkv, d, T, ctx, page = (c[k] for k in ("B", "H", "Hkv", "d", "T", "ctx", "page"))
        s["X"] = r.normal(B, T, H * d)
        s["W_r"], s["b_r"] = _router_weights(r, H * d)
        s["Q"] = r.normal(B, H, T, d)
        s["newK"], s["newV"] = ([r.normal(B, Hkv, T, d) for _ in range(3)] for _ in range(2))
        s["n"] = (ctx + T, ctx + T, c["n3"])
        s["pk"], s["pv"], s["tab"] = zip(*(_pool(r, B, Hkv, m, page, d) for m in s["n"]))
        s["shape"] = mka.make_shape(B, H, T, d, D=H * d, window=c["W"], q_offset=ctx)
        s["ws"] = torch.zeros(256, dtype=torch.uint8, device=_DEV)
    elif kind == "decode":
        B, H, Hkv, d = (c[k] for k in ("B", "H", "Hkv", "d"))
        s["X"] = r.normal(B, H * d)
        s["W_r"], s["b_r"] = _router_weights(r, H * d)
        s["q"] = r.normal(B, H, d)
        n = (c["n1"], c["n2"], c["n3"])
        s["K"] = [r.normal(B, Hkv, m, d) for m in n]
        s["V"] = [r.normal(B, Hkv, m, d) for m in n]
        s["shape"] = mka.make_shape(B, H, 1, d, D=H * d, kv_heads=Hkv)
        s["ws"] = mka.alloc_workspace(s["shape"], n, mka.MKA_WS_DECODE, _DEV)
        s["gate"] = torch.empty(B, 3, dtype=_F32, device=_DEV)
        s["O"], s["LSE"] = torch.empty_like(s["q"]), torch.empty(B, H, dtype=_F32, device=_DEV)
    elif kind == "serve":
        B, H, Hkv, d, page, bank, R = (c[k] for k in ("B", "H", "Hkv", "d", "page", "bank", "R"))
        s["X"] = r.normal(B, 1, H * d)
        s["W_r"], s["b_r"] = _router_weights(r, H * d)
        s["q"] = r.normal(B, H, d)
        s["newK"], s["newV"] = ([r.normal(B, Hkv, 1, d) for _ in range(3)] for _ in range(2))
        s["n"] = (c["n1"], c["n2"], R * page)
        k1, v1, t1 = _pool(r, B, Hkv, c["n1"], page, d)
        k2, v2, t2 = _pool(r, B, Hkv, c["n2"], page, d)
        k3, v3, bank_tab = _pool(r, B, Hkv, bank * page, page, d)
        s["pk"], s["pv"], s["t1"], s["t2"], s["bank"] = (k1, k2, k3), (v1, v2, v3), t1, t2, bank_tab
        len2 = _lengths(B, c["n2"])
        s["rows1"] = torch.tensor([min(c["n1"], m) for m in len2], dtype=torch.int32, device=_DEV)
        s["rows2"] = torch.tensor(len2, dtype=torch.int32, device=_DEV)
        s["at"] = s["rows2"] - 1                                         # the new token's row
        s["bank_len"] = torch.tensor(_lengths(B, bank), dtype=torch.int32, device=_DEV)
        s["proj"] = r.normal(c["bits"], d, dtype=_F32)
        s["codes"] = mka.mka_l3_index(k3, s["proj"])
        s["shape"] = mka.make_shape(B, H, 1, d, D=H * d)
        s["ws"] = torch.empty(mka.mka_decode_paged_workspace_bytes(s["shape"], Hkv, s["n"]), dtype=torch.uint8, device=_DEV)
        s["gate"] = torch.empty(B, 1, 3, dtype=_F32, device=_DEV)
        s["t3"] = torch.empty(B, Hkv, R, dtype=torch.int32, device=_DEV)
        s["n_sel"], s["rows3"] = (torch.empty(B, dtype=torch.int32, device=_DEV) for _ in range(2))
        s["O"], s["LSE"] = torch.empty_like(s["q"]), torch.empty(B, H, dtype=_F32, device=_DEV)
    elif kind == "summary":
        B, T, D = c["B"], c["T"], c["D"]
        s["X"] = r.normal(B, T, D, dtype=_BF16 if c["bf16"] else _F32)
        s["state"] = r.normal(B, D, dtype=_F32)
        s["ws"] = mka.mka_l2_summary_workspace(s["X"])
        s["M2"] = torch.empty_like(s["X"])
    elif kind == "index":
        s["pool"] = r.normal(c["pages"], c["Hkv"], c["page"], c["d"])
        s["proj"] = r.normal(c["bits"], c["d"], dtype=_F32)
        s["codes"] = torch.empty(c["pages"], c["Hkv"], c["bits"] // 32, dtype=torch.int32, device=_DEV)
    else:
        raise ValueError(kind)
    return s


def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind in ("train", "fp32"):
        gate = mka.mka_router(s["X"], s["W_r"], s["b_r"])
        O, LSE = mka.mka_fwd(s["shape"], s["Q"], s["K"], s["V"], gate, ws=s["ws"])
        g = mka.mka_bwd(s["shape"], s["Q"], s["K"], s["V"], gate, O, LSE, s["dO"], R=s["X"], ws=s["ws_bwd"])
        out = [gate, O, LSE, g["dQ"], g["dK"], g["dV"], g["dG"], g["dW_r"], g["db_r"]]
        if kind == "fp32":
            out.append(mka.mka_fwd(s["shape_full"], s["Q"], s["K"], s["V"], gate, ws=s["ws"])[0])
        return out
    if kind == "prefill":
        gate = mka.mka_router(s["X"], s["W_r"], s["b_r"])
        return [gate, *mka.mka_fwd(s["shape"], s["Q"], s["K"], s["V"], gate, ws=s["ws"])]
    if kind == "chunk":
        gate = mka.mka_router(s["X"], s["W_r"], s["b_r"])
        mka.mka_fuse_kv_paged(s["newK"], s["newV"], gate, s["pk"][1], s["pv"][1], s["tab"][1], dst_offset=c["ctx"])
        O, LSE = mka.mka_fwd_paged(s["shape"], c["Hkv"], s["Q"], s["pk"], s["pv"], s["tab"], s["n"], gate, ws=s["ws"])
        return [gate, O, LSE, s["pk"][1], s["pv"][1]]
    if kind == "decode":
        mka.mka_router(s["X"], s["W_r"], s["b_r"], gate=s["gate"])
        mka.mka_decode(s["shape"], s["q"], s["K"], s["V"], s["gate"], O=s["O"], LSE=s["LSE"], ws=s["ws"])
        return [s["gate"], s["O"], s["LSE"]]
    if kind == "serve":
        mka.mka_router(s["X"], s["W_r"], s["b_r"], gate=s["gate"])
        mka.mka_fuse_kv_paged(s["newK"], s["newV"], s["gate"], s["pk"][1], s["pv"][1], s["t2"], dst_offsets=s["at"])
        mka.mka_l3_retrieve(s["q"], c["Hkv"], s["proj"], s["codes"], s["bank"], s["bank_len"], c["R"], c["page"], table=s["t3"],
                            n_sel=s["n_sel"], rows=s["rows3"])
        mka.mka_decode_paged(s["shape"], c["Hkv"], s["q"], s["pk"], s["pv"], (s["t1"], s["t2"], s["t3"]), s["n"], s["gate"].view(-1, 3),
                             rows=(s["rows1"], s["rows2"], s["rows3"]), O=s["O"], LSE=s["LSE"], ws=s["ws"])
        return [s["gate"], s["pk"][1], s["pv"][1], s["t3"], s["n_sel"], s["rows3"], s["O"], s["LSE"]]
    if kind == "summary":
        # a carried EMA session is read as it was left; a fresh session only writes its state
        M2 = mka.mka_l2_summary(s["X"], kind=mka.MKA_SUMMARY_EMA if c["ema"] else mka.MKA_SUMMARY_MEAN, beta=0.9, state=s["state"],
                                n_prev=1000 if c["carry"] else 0, M2=s["M2"], ws=s["ws"])
        return [M2, s["state"]]
    return [mka.mka_l3_index(s["pool"], s["proj"], codes=s["codes"])]


def _pairs(T, W, n1, n2, n3, ctx=0):
    """Visible (query, key) pairs of one head: window, causal prefix and every long-term slot."""
    p0, p1 = ctx, ctx + T - 1
    full = sum(min(p + 1, W) for p in range(p0, min(p1, W) + 1)) + W * max(0, p1 - max(p0, W + 1) + 1)
    return full + (p0 + 1 + p1 + 1) * T // 2 + T * n3


def work(case):
    c = case
    kind = c["kind"]
    if kind in ("train", "fp32", "prefill", "chunk"):
        B, H, d, T = c["B"], c["H"], c["d"], c["T"]
        Hkv = c.get("Hkv", H)
        es = 4 if kind == "fp32" else 2
        ctx = c.get("ctx", 0)
        n = (ctx + T, ctx + T, c["n3"])
        pairs = _pairs(T, c["W"], *n, ctx=ctx) * B * H
        # rows of the window level that some query sees
        rows = min(n[0], T + c["W"] - 1) + n[1] + n[2]
        q_bytes, kv_bytes = B * H * T * d * es, 2 * B * Hkv * rows * d * es
        nbytes = B * T * H * d * es + 2 * q_bytes + kv_bytes
        flops = 4.0 * d * pairs
        if kind in ("train", "fp32"):                                    # dO in, dQ, dK, dV out
            nbytes += 2 * q_bytes + kv_bytes
            flops += 10.0 * d * pairs
        if kind == "fp32":                                               # the second form of the forward
            nbytes += q_bytes
            flops += 4.0 * d * pairs
        if kind == "chunk":                                              # three levels in, the fused rows out
            nbytes += 8 * B * Hkv * T * d * es
        return {"bytes": nbytes, "flops": flops}
    if kind == "decode":
        rows = c["B"] * (c["n1"] + c["n2"] + c["n3"])
        return {"bytes": 4 * rows * c["Hkv"] * c["d"] + 2 * c["B"] * c["H"] * c["d"] * 3, "flops": 4.0 * rows * c["H"] * c["d"]}
    if kind == "serve":
        len2 = _lengths(c["B"], c["n2"])
        chunks = _lengths(c["B"], c["bank"])
        rows = sum(m + min(c["n1"], m) for m in len2) + sum(min(c["R"], m) * c["page"] for m in chunks)
        codes = sum(chunks) * (c["bits"] // 8 * c["Hkv"] + 4)
        return {"bytes": 4 * rows * c["Hkv"] * c["d"] + codes + 2 * c["B"] * c["H"] * c["d"] * 3, "flops": 4.0 * rows * c["H"] * c["d"]}
    if kind == "summary":
        return {"bytes": 2 * c["B"] * c["T"] * c["D"] * (2 if c["bf16"] else 4), "flops": 3.0 * c["B"] * c["T"] * c["D"]}
    keys = c["pages"] * c["Hkv"] * c["page"]
    return {"bytes": 2 * keys * c["d"] + c["pages"] * c["Hkv"] * c["bits"] // 8,
            "flops": keys * c["d"] + 2.0 * c["pages"] * c["Hkv"] * c["bits"] * c["d"]}


def tolerance(case):
    """About four times what the tensor-core kernels differ from the CUDA-core ones and from 64-bit arithmetic by."""
    kind = case["kind"]
    if kind == "index":                                                  # code bits are decided in a fixed order
        return "exact"
    if kind == "fp32":                                                   # measured: 8e-7, single values 1.3e-5
        return {"rel": 4e-6, "max": 5e-5}
    if kind == "summary":                                                # bf16: the one rounding; fp32: 2e-7, 2.4e-6
        return {"rel": 4e-3, "max": 1.6e-2} if case["bf16"] else {"rel": 1e-6, "max": 1e-5}
    if kind == "train":                                                  # gradients: 3.3e-3, single values 3.1e-2
        return {"rel": 1.2e-2, "max": 0.12}
    return {"rel": 1e-2, "max": 7e-2}                                    # outputs: 2.5e-3, 1.8e-2


def _softmax_parts(s, b, h, i0, i1, gate, K, V, ctx):
    """Gated scores of query rows [i0, i1) of one head in 64 bits: per level (first key, scores + log gate, keys, values)."""
    c = s["case"]
    T, d, W = c["T"], c["d"], c["W"]
    q = s["Q"][b, h, i0:i1].double() * d ** -0.5
    p = torch.arange(ctx + i0, ctx + i1, device=_DEV)[:, None]
    out = []
    for l in range(3):
        lo = max(0, ctx + i0 - W + 1) if l == 0 else 0
        hi = min(K[l].shape[0], ctx + i1) if l < 2 else K[l].shape[0]
        k, v = K[l][lo:hi], V[l][lo:hi]
        x = q @ k.T + torch.log(gate[b, i0:i1, l:l + 1])
        if l < 2:
            j = torch.arange(lo, hi, device=_DEV)[None]
            x.masked_fill_((j > p) | (j <= p - W) if l == 0 else j > p, float("-inf"))
        out.append((lo, x, k, v))
    return out


def _attention64(s, gate, head_kv, ctx=0, dO=None, full=False, rows=1024):
    """Forward (and, with dO, backward) in 64 bits, one head and some query rows at a time."""
    c = s["case"]
    B, H, T, d = c["B"], c["H"], c["T"], c["d"]
    new = lambda *n: torch.zeros(*n, dtype=torch.float64, device=_DEV)  # noqa: E731
    O, LSE, F = new(B, H, T, d), new(B, H, T), new(B, H, T, d) if full else None
    if dO is not None:
        dQ, dG = new(B, H, T, d), new(B, T, 3)
        dK, dV = ([new(*k.shape) for k in s["K"]] for _ in range(2))
    for b in range(B):
        for h in range(H):
            g = h // (H // c.get("Hkv", H))
            K, V = head_kv(b, g)
            for i0 in range(0, T, rows):
                i1 = min(T, i0 + rows)
                parts = _softmax_parts(s, b, h, i0, i1, gate, K, V, ctx)
                if full:
                    F[b, h, i0:i1] = sum(gate[b, i0:i1, l:l + 1] * (torch.softmax(x, 1) @ v) for l, (_, x, _, v) in enumerate(parts))
                lse = torch.logsumexp(torch.stack([torch.logsumexp(x, 1) for _, x, _, _ in parts]), 0)
                P = [x.sub_(lse[:, None]).exp_() for _, x, _, _ in parts]
                o = sum(pl @ v for pl, (_, _, _, v) in zip(P, parts))
                O[b, h, i0:i1], LSE[b, h, i0:i1] = o, lse
                if dO is None:
                    continue
                do, q = dO[b, h, i0:i1].double(), s["Q"][b, h, i0:i1].double()
                for l, (pl, (lo, _, k, v)) in enumerate(zip(P, parts)):
                    at = slice(lo, lo + k.shape[0])
                    dV[l][b, g, at] += pl.T @ do
                    ds = pl.mul_(do @ v.T - (do * o).sum(1, keepdim=True))
                    dG[b, i0:i1, l] += ds.sum(1)
                    dQ[b, h, i0:i1] += (ds @ k) * d ** -0.5
                    dK[l][b, g, at] += (ds.T @ q) * d ** -0.5
    if dO is not None:
        x = s["X"].double().reshape(-1, H * d)
        return O, LSE, F, dQ, dK, dV, dG, x.T @ dG.view(-1, 3), dG.view(-1, 3).sum(0)
    return O, LSE


def exact(case, seed):
    """The outputs of ``run`` in 64 bits, from torch alone (``prepare`` gives the inputs)."""
    if case["kind"] == "index":                                          # code bits, not numbers
        return None
    s = prepare(case, seed)
    c = s["case"]
    kind = c["kind"]
    if kind == "summary":
        X, M2, step = s["X"], torch.empty(s["X"].shape, dtype=torch.float64, device=_DEV), 256
        m = s["state"].double() if c["carry"] else X[:, 0].double() if c["ema"] else torch.zeros_like(s["state"], dtype=torch.float64)
        i = torch.arange(step, device=_DEV, dtype=torch.float64)
        keep = float(torch.tensor(0.9, dtype=_F32))                      # the call takes its decay in 32 bits
        decay = torch.where(i[:, None] >= i[None], keep ** (i[:, None] - i[None]).clamp_min(0), 0.0) * (1.0 - keep if c["ema"] else 0.0)
        for t in range(0, X.shape[1], step):
            x = X[:, t:t + step].double()
            n = x.shape[1]
            if c["ema"]:
                y = decay[:n, :n] @ x + keep ** (i[:n, None] + 1) * m[:, None]
                M2[:, t:t + n] = y
            else:
                y = x.cumsum(1) + m[:, None]
                M2[:, t:t + n] = y / (t + 1 + i[:n, None])
            m = y[:, -1]
        return [M2, m]
    gate = torch.softmax(s["X"].double() @ s["W_r"].double() + s["b_r"].double(), -1)
    if kind in ("train", "fp32", "prefill"):
        kv = lambda b, g: ([x[b, g].double() for x in s["K"]], [x[b, g].double() for x in s["V"]])  # noqa: E731
        if kind == "prefill":
            return [gate, *_attention64(s, gate, kv)]
        O, LSE, F, dQ, dK, dV, dG, dW, db = _attention64(s, gate, kv, dO=s["dO"], full=kind == "fp32")
        return [gate, O, LSE, dQ, dK, dV, dG, dW, db] + ([F] if kind == "fp32" else [])
    if kind == "decode":
        O, LSE = torch.empty(s["q"].shape, dtype=torch.float64, device=_DEV), torch.empty(c["B"], c["H"], dtype=torch.float64, device=_DEV)
        for b in range(c["B"]):
            q = s["q"][b].double().view(c["Hkv"], -1, c["d"]) * c["d"] ** -0.5
            x = torch.cat([q @ k[b].double().transpose(1, 2) + torch.log(gate[b, l]) for l, k in enumerate(s["K"])], 2)
            LSE[b] = torch.logsumexp(x, 2).view(-1)
            O[b] = (torch.softmax(x, 2) @ torch.cat([v[b].double() for v in s["V"]], 1)).view(c["H"], c["d"])
        return [gate, O, LSE]
    # chunk and serve: the fused rows in the session pool
    pools = []
    at = s["at"].long() if kind == "serve" else torch.full((c["B"],), c["ctx"], device=_DEV)
    tab = (s["t2"] if kind == "serve" else s["tab"][1]).long()
    for pool, new in ((s["pk"][1], s["newK"]), (s["pv"][1], s["newV"])):
        pool = pool.double()
        for b in range(c["B"]):
            r = at[b] + torch.arange(new[0].shape[2], device=_DEV)
            pool[tab[b, r // c["page"]], :, r % c["page"]] = sum(gate[b, :, l, None] * x[b].double() for l, x in enumerate(new)).transpose(0, 1)
        pools.append(pool)
    if kind == "serve":                                                  # what is recalled hangs on single code bits
        return [gate, *pools, None, None, None, None, None]

    def paged(b, g):
        out = []
        for src, fused in ((s["pk"], pools[0]), (s["pv"], pools[1])):
            out.append([(fused.to(_BF16) if l == 1 else src[l])[s["tab"][l][b].long(), g].reshape(-1, c["d"])[:s["n"][l]].double() for l in range(3)])
        return out

    return [gate, *_attention64(s, gate, paged, ctx=c["ctx"]), *pools]

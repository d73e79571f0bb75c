// Tensor-core backward of Eq. 5 for bf16 on sm_100a: TMA -> shared memory -> tcgen05.mma -> TMEM.
//
// The paper prints no backward; this one follows from differentiating Eq. 5.  With
//   p = lambda_{t,l} exp(s - LSE_t) on the visible set,  dP = dO_t . v_{l,j},  D_t = dO_t . O_t,
//   dS = p (dP - D_t):
//     dV_{l,j} = sum_t p dO_t      dK_{l,j} = tau sum_t dS q_t      dQ_t = tau sum_{l,j} dS k_{l,j}
//     G_{t,l}  = sum_{j in l} dS   (gradient of the router logit of level l, per head)
//
// Three launches, each deterministic (every output element has one owner, fixed summation order):
//   bwd_prep_kernel    per (b,h,t): D_t and, per level, the exponent bias log2(lambda) - LSE log2(e)
//   bwd_dq_tc_kernel   CTA = 128 query rows of one (b,h); streams the level-ordered list of 128-row
//                      key tiles (L1 window, L2 prefix, L3 slots) exactly like the forward:
//                      S = Q K^T, dP = dO V^T (128x128 each), dS -> TMEM (bf16), dQ += dS K.
//   bwd_dkv_tc_kernel  CTA = 128 key rows of one level of one (b,h); streams the 128-row query
//                      tiles that can see them: S^T = K Q^T, dP^T = V dO^T, P^T and dS^T -> TMEM
//                      (bf16), dV += P^T dO, dK += dS^T Q.
// Both kernels recompute the scores (7 matrix products per visible tile pair instead of 5) in exchange
// for needing no atomics and no cross-CTA reduction.
//
// In the dK/dV kernel the per-query terms vary along the COLUMNS of the transposed tiles, where a thread would need 64
// biases and 64 D_t per tile from shared memory (which the tensor pipe saturates).  They enter through the tensor pipe
// instead: both score products get a ninth K-step whose key-side operand is ones and whose query-side operand holds
// bias_t / scale (for S^T) or -D_t (for dP^T), each split into three bf16 terms, so S^T + bias / scale and dP^T - D arrive
// in TMEM ready-made.  Two warps of their own write those 4 KB operand slabs (no swizzle) from the statistics of the prep
// kernel, fetched one tile ahead.  Q tiles and dO tiles travel in rings of their own: dO(e) is free again after dV(e),
// Q(e) only after dK(e), and Q(e+1) is what the next score product waits for.  At d = 128 a quarter of the exponentials of that
// kernel run as a cubic on the FMA pipe (exp2_pair_fma).
//
// CTAs are persistent: they take output tiles (items) from a ticket counter, and the next item's copies and first products run
// under the element-wise threads' stores of the previous one.
//
// Warp roles: the first eight warps (d = 64: sixteen) are the element-wise ("softmax") threads: thread i of a
// warpgroup owns TMEM lane i & 127 (a query row in the dQ kernel, a key row in the dK/dV kernel) and the
// warpgroup's share of a tile's columns (64, d = 64: 32).  Their work on a tile has
// two phases so that it overlaps the tensor pipe: phase 1 needs only S (p = 2^(s*scale + bias), kept in
// registers) and runs while dP is still being multiplied; phase 2 reads dP, forms dS = p (dP - D) and
// writes it (bf16) over the columns of dP it has just read.  The next warp issues the TMA loads; the one
// after it issues every tcgen05.mma, running its loop converged with one elected lane issuing; two more write the slabs (dK/dV).
// TMEM (512 columns), dQ kernel: S ping [0,128), S pong [128,256), dP/dS [256,384), dQ [384,384+d).
//                     dK/dV kernel: S^T/P^T [0,128), dP^T/dS^T [128,256), dK [256,256+d), dV [256+d,256+2d), d = 64: second S^T [384,512).
// Every mbarrier wait is bounded; on expiry the CTA raises a flag, drains and reports MKA_ERR_TIMEOUT.
#include "tc_ptx.cuh"

namespace mka {
namespace {

constexpr int kBlk = 128;                             // rows of every tile
constexpr uint32_t kPanel = 128 * 128;                // bytes of a [128 rows][64 bf16] panel
constexpr int kMaxStages = 4;

struct BwdMaps {
    CUtensorMap q, dO;
    CUtensorMap k[3], v[3];
};

struct BwdTcParams {
    __nv_bfloat16* dQ;
    const float* statD;       // [B*H, Tpad]  D_t = dO_t . O_t
    const float* statB[3];    // per level: [B*H, Tpad]  log2(lambda_{t,l}) - LSE_t log2(e)  (-inf on padding rows)
    float* Gpart;             // [B, H, T, 3]
    LevelGradDev dL[3];
    long long n[3];
    int B, H, T, Tpad;
    int kv_group;             // query heads per KV head: K, V, dK, dV hold H / kv_group heads
    int window, q_offset;
    float scale, scale_log2;
    int kv_tiles[3];          // 128-row key tiles per level
    int H_kv;
    long long dkv_items;      // key tiles of all levels, KV heads and batches
    long long dq_items;       // query tiles of all heads and batches
    unsigned int *dkv_ticket, *dq_ticket, *gate_ticket;   // zero at launch
    float* dG;                // null: not the dK/dV kernel's
    int dq_first, in_place;   // order of the two kernels (see launch_t); a gradient of keys or values is written over keys or values
    unsigned int* status;
    unsigned long long wait_limit_ns;
    int test_stall;           // test hook: the dK/dV kernel's loader leaves out the last query tile of every CTA
};

// v as a sum of three bf16 terms (exact to 2^-25 |v|) in the first three of eight bf16 slots of a 16-byte core-matrix row;
// an infinite v (the bias of a padding row or of a level the gate closes) stays one infinite term.
__device__ __forceinline__ uint4 split3_bf16(float v) {
    if (!(fabsf(v) <= 3.0e38f)) return make_uint4(pack_bf16(v, 0.f), 0u, 0u, 0u);
    const float t0 = __bfloat162float(__float2bfloat16_rn(v));
    const float r1 = v - t0;
    const float t1 = __bfloat162float(__float2bfloat16_rn(r1));
    return make_uint4(pack_bf16(t0, t1), pack_bf16(r1 - t1, 0.f), 0u, 0u);
}

// 2^x for two arguments x <= 0 on the FMA pipe: x is clamped to -127 and split into n = round(x) and f = x - n in
// [-1/2, 1/2] by adding and subtracting 1.5 * 2^23 (the sum's low mantissa bits are n); 2^f is a cubic with constant term
// exactly 1 (coefficients fitted for the smallest maximum relative error, 1.0e-4, a twentieth of the rounding step of
// the bf16 value it becomes); n is added to the exponent field.  x <= -127 gives exactly 0, as ex2 does for -inf.
__device__ __forceinline__ void exp2_pair_fma(float x0, float x1, float& p0, float& p1) {
    const float kMagic = 12582912.f;
    const uint64_t x = pack2(fmaxf(x0, -127.f), fmaxf(x1, -127.f));
    const uint64_t t = add2(x, pack2(kMagic, kMagic));
    const uint64_t n = add2(t, pack2(-kMagic, -kMagic));
    const uint64_t f = fma2(n, pack2(-1.f, -1.f), x);
    uint64_t r = fma2(pack2(0.05500893f, 0.05500893f), f, pack2(0.24221095f, 0.24221095f));
    r = fma2(r, f, pack2(0.69328290f, 0.69328290f));
    r = fma2(r, f, pack2(1.f, 1.f));
    float r0, r1, t0, t1;
    unpack2(r, r0, r1);
    unpack2(t, t0, t1);
    p0 = __uint_as_float(__float_as_uint(r0) + (__float_as_uint(t0) << 23));
    p1 = __uint_as_float(__float_as_uint(r1) + (__float_as_uint(t1) << 23));
}

template <int DH>
struct BCfg {
    static constexpr int kEw = DH == 128 ? 8 : 16;                    // element-wise warps
    static constexpr int kGroups = kEw / 4;                   // threads per row: warpgroup w owns columns [w * kCols, (w + 1) * kCols) of a tile
    static constexpr int kCols = kBlk / kGroups;
    static constexpr int kProducerWarp = kEw, kMmaWarp = kEw + 1;
    static constexpr int kSlabWarp = kEw + 2;                 // dK/dV kernel: this one and the next write the operand slabs
    static constexpr int kThreads = (kEw + 2) * 32, kThreadsDkv = (kEw + 4) * 32;
    // A-operand column (32-bit TMEM columns) of K-step k of a 128-wide bf16 row: every warpgroup packs its kCols columns into
    // the first kCols / 2 of the TMEM columns it has read them from.  The weights are handed over in two parts, the first and
    // the second half of every thread's columns: K-step kstep(part, i), i = 0..3.
    static __host__ __device__ constexpr uint32_t packed_col(int k) { return (uint32_t)((k * 16 / kCols) * kCols + (k * 16 % kCols) / 2); }
    static __host__ __device__ constexpr int kstep(int part, int i) { return kGroups == 2 ? (i >> 1) * 4 + part * 2 + (i & 1) : 2 * i + part; }
    static constexpr int kGsm = DH == 128 ? 1 : kGroups - 1;  // warpgroups whose row sums meet in shared memory at a time (dQ kernel)
    static constexpr int kPanels = DH / 64;
    static constexpr uint32_t kTile = kPanels * kPanel;       // a 128-row tile
    static constexpr int kStages = DH == 128 ? 2 : 4;         // also keeps the CTA above half of shared memory
    // dK/dV kernel: the per-query terms enter the two score products as one more K-step (see kAugBytes below)
    static constexpr uint32_t kAugBytes = kBlk * 16 * 2;              // a [128 rows][16] bf16 operand slab without swizzle
    static constexpr int kStagesK = DH == 128 ? 3 : 4;        // K ring of the dQ kernel: K(e) stays in use until dQ(e), two tiles after it is first read
    static constexpr uint32_t kSmemDq = 2 * kTile + (kStages + kStagesK) * kTile + 1024;
    static constexpr uint32_t kSmemDkv = 2 * kTile + kStages * (2 * kTile + 2 * kAugBytes) + kAugBytes + 1024;
    // instruction descriptors: fp32 accumulate, bf16 x bf16, M = 128
    static constexpr uint32_t kIdescS = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kBlk >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
    static constexpr uint32_t kIdescAcc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((uint32_t)(DH >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
};

struct BwdBarriers {
    uint64_t fixed_full;                                  // the CTA's own (non-streamed) tiles
    uint64_t a_full[kMaxStages], a_empty[kMaxStages];     // streamed ring (dQ kernel: K tiles; dK/dV kernel: Q tiles + bias slabs)
    uint64_t b_full[kMaxStages], b_empty[kMaxStages];     // second streamed ring (dQ kernel: V tiles; dK/dV kernel: dO tiles + D slabs)
    uint64_t s_full[2];                                   // S landed in TMEM (dQ kernel: ping, pong)
    uint64_t dp_full;                                     // dP landed in TMEM
    uint64_t p_part[2];                                   // phase 1 (dK/dV kernel): the first / second half of every thread's P^T columns is written; with two S^T: all of the P^T over S^T buffer 0 / 1
    uint64_t ds_part[2];                                  // phase 2: the same for dS
    uint64_t acc_done;                                    // per item: its accumulators are complete
    uint64_t fixed_free;                                  // per item: its own tiles have had their last reader
    uint64_t item_full[2], item_free[2];                  // the item numbers, two slots
};

// Which of two barriers completes first (0 or 1; the first one when both have), -1 when the wait was given up.  Executed by a
// converged warp; bounded like every other wait.
__device__ __forceinline__ int poll_two(uint64_t* b0, uint32_t ph0, uint64_t* b1, uint32_t ph1, volatile WaitCtl* ctl) {
    int got = -2;
    if (__all_sync(0xffffffffu, mbar_try(b0, ph0))) return 0;
    if (__all_sync(0xffffffffu, mbar_try(b1, ph1))) return 1;
    const unsigned long long t0 = gtimer();
    while (got == -2) {
        if (__all_sync(0xffffffffu, mbar_try(b0, ph0))) got = 0;
        else if (__all_sync(0xffffffffu, mbar_try(b1, ph1))) got = 1;
        else {
            bool give_up = ctl->abort != 0;
            if (!give_up && gtimer() - t0 > ctl->limit_ns) { ctl->abort = 1; give_up = true; }
            if (__any_sync(0xffffffffu, give_up)) got = -1;
        }
    }
    return __shfl_sync(0xffffffffu, got, 0);
}

// Items (output tiles) are dealt from a ticket counter: a CTA takes the next one when it is free, in the order in which
// blocks of a plain grid would start.  The producing warp posts the number of item `it` to the other roles; a number past
// the last item ends them all.
// The posted item is the whole description (Item: ints only), so that its divisions are made once and early.
template <typename Item>
__device__ __forceinline__ bool post_item(BwdBarriers& bar, Item (&items)[2], int it, const Item& item, int lane, volatile WaitCtl* ctl) {
    if (it >= 2 && !mbar_wait_warp(&bar.item_free[it & 1], (uint32_t)((it >> 1) - 1) & 1u, ctl)) return false;
    if (lane == 0) {
        items[it & 1] = item;
        mbar_arrive(&bar.item_full[it & 1]);
    }
    __syncwarp();
    return true;
}
template <typename Item>
__device__ __forceinline__ bool take_item(BwdBarriers& bar, Item (&items)[2], int it, Item& item, int lane, volatile WaitCtl* ctl) {
    if (!mbar_wait_warp(&bar.item_full[it & 1], (uint32_t)(it >> 1) & 1u, ctl)) return false;
    const int* src = reinterpret_cast<const int*>(&items[it & 1]);
    int v[sizeof(Item) / 4];
#pragma unroll
    for (int i = 0; i < (int)(sizeof(Item) / 4); ++i) v[i] = __shfl_sync(0xffffffffu, src[i], 0);      // warp-uniform for the compiler too
    memcpy(&item, v, sizeof(Item));
    __syncwarp();
    if (lane == 0) mbar_arrive(&bar.item_free[it & 1]);
    return true;
}

template <int kWarps> __device__ __forceinline__ void softmax_group_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kWarps * 32) : "memory"); }
template <int kWarps> __device__ __forceinline__ bool softmax_group_all(bool flag) {        // the same barrier; true when it is for all of its threads
    uint32_t out;
    asm volatile("{\n.reg .pred pi, po;\nsetp.ne.u32 pi, %1, 0;\nbar.red.and.pred po, 1, %2, pi;\nselp.u32 %0, 1, 0, po;\n}"
                 : "=r"(out) : "r"((uint32_t)flag), "n"(kWarps * 32) : "memory");
    return out != 0;
}

// ------------------------------------------------------------------------------------------ prep
// D = dO . O and the three exponent biases of every padded row.  DH / 8 lanes share a row (one 16-byte load of O and
// one of dO each), a warp covers 2 or 4 rows per pass and a thread works on four passes at once, so eight loads are
// in flight per thread; the row's LSE and gate are fetched with them.  blockIdx.y is the (batch, head): with the row split
// by 64-bit divisions the arithmetic took most of the time (2.5 TB/s).  Each lane finishes one row: with the row's first lane
// loading and storing for it, two rows at a time, the pass took 82 us at [4, 16, 8192, 128] and 19 us at [8, 16, 2048, 64],
// now 53 and 16 (62 registers before, 37 now).  Padding rows (t >= T) get a bias of -inf so
// that a streamed sub-tile may run past the last query without a mask.
template <int DH>
__global__ void __launch_bounds__(256) bwd_prep_kernel(const __nv_bfloat16* __restrict__ O, const __nv_bfloat16* __restrict__ dO,
                                                       const float* __restrict__ LSE, const float* __restrict__ gate, int H,
                                                       int T, int Tpad, float* __restrict__ sD,
                                                       float* __restrict__ b0, float* __restrict__ b1, float* __restrict__ b2,
                                                       unsigned int* __restrict__ header) {
    chain_enter();
    if (threadIdx.x < 4 && (blockIdx.x | blockIdx.y | blockIdx.z) == 0) header[threadIdx.x] = 0u;   // status word and tickets of the kernels that follow
    constexpr int LPR = DH / 8;                            // lanes per row: 16 or 8
    constexpr int RPW = 32 / LPR;                          // rows per warp and pass
    constexpr int kPasses = 4, kRows = RPW * kPasses;      // rows of a warp: 8 or 16
    const int lane = threadIdx.x & 31, sub = lane % LPR, grp = lane / LPR;
    const long long bh = (long long)blockIdx.z * H + blockIdx.y;
    const int row0 = (blockIdx.x * 8 + (threadIdx.x >> 5)) * kRows;
    const __nv_bfloat16* Ob = O + bh * T * DH + sub * 8;
    const __nv_bfloat16* dOb = dO + bh * T * DH + sub * 8;
    uint4 a[kPasses], g[kPasses];
#pragma unroll
    for (int u = 0; u < kPasses; ++u) {
        const int t = row0 + u * RPW + grp;
        a[u] = g[u] = make_uint4(0u, 0u, 0u, 0u);
        if (t < T) {
            a[u] = __ldg(reinterpret_cast<const uint4*>(Ob + (long long)t * DH));
            g[u] = __ldg(reinterpret_cast<const uint4*>(dOb + (long long)t * DH));
        }
    }
    // lane i < kRows finishes row i of the warp: its LSE and gate on the way in, its four values on the way out, are then
    // consecutive in memory (by the row's first lane, pass by pass, they were 32 accesses of two rows each)
    const int t_own = row0 + lane;
    float lse = -INFINITY, gt[3] = {0.f, 0.f, 0.f}, own = 0.f;
    if (lane < kRows && t_own < T) {
        lse = LSE[bh * T + t_own];
        const float* gr = gate + ((long long)blockIdx.z * T + t_own) * 3;
        gt[0] = gr[0]; gt[1] = gr[1]; gt[2] = gr[2];
    }
#pragma unroll
    for (int u = 0; u < kPasses; ++u) {
        const uint32_t aw[4] = {a[u].x, a[u].y, a[u].z, a[u].w}, gw[4] = {g[u].x, g[u].y, g[u].z, g[u].w};
        float s = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            s = fmaf(__uint_as_float(aw[i] << 16), __uint_as_float(gw[i] << 16), s);
            s = fmaf(__uint_as_float(aw[i] & 0xffff0000u), __uint_as_float(gw[i] & 0xffff0000u), s);
        }
#pragma unroll
        for (int o = LPR / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        const float of_row = __shfl_sync(0xffffffffu, s, (lane % RPW) * LPR);
        if (lane / RPW == u) own = of_row;
    }
    if (lane < kRows && t_own < Tpad) {
        const bool live = lse > -INFINITY;
        const float l2 = lse * kLog2e;
        const long long at = bh * Tpad + t_own;
        sD[at] = own;
        b0[at] = (live && gt[0] > 0.f) ? log2f(gt[0]) - l2 : -INFINITY;
        b1[at] = (live && gt[1] > 0.f) ? log2f(gt[1]) - l2 : -INFINITY;
        b2[at] = (live && gt[2] > 0.f) ? log2f(gt[2]) - l2 : -INFINITY;
    }
}

// Scores outside columns [c_lo, c_hi) of the thread's become -inf: one bit per column, so a column costs a test and a
// select; 32 columns that no row of the warp masks are passed over.
template <int N>
__device__ __forceinline__ void mask_cols(float (&x)[N], int c_lo, int c_hi) {
#pragma unroll
    for (int c0 = 0; c0 < N; c0 += 32) {
        const uint32_t vis = low_bits(c_hi - c0) & ~low_bits(c_lo - c0);
        if (__all_sync(0xffffffffu, vis == 0xffffffffu)) continue;
#pragma unroll
        for (int i = 0; i < 32; ++i) x[c0 + i] = (vis >> i) & 1u ? x[c0 + i] : -INFINITY;
    }
}

// Key tile range [first, end) (128-row units) of query rows [r0, r1] on one level.
__device__ __forceinline__ void key_tile_range(int level, long long r0, long long r1, int q_offset, int window, long long n,
                                               int& first, int& end) {
    long long lo_f, hi_f, lo_l, hi_l;
    visible_range(level, r0 + q_offset, window, n, 0, lo_f, hi_f);
    visible_range(level, r1 + q_offset, window, n, 0, lo_l, hi_l);
    const long long hi = hi_l > hi_f ? hi_l : hi_f;
    if (hi <= lo_f) { first = end = 0; return; }
    first = (int)(lo_f / kBlk);
    end = (int)((hi + kBlk - 1) / kBlk);
}

// N 32-bit TMEM columns of this thread's lane, N = 16 or a multiple of 32.
template <int N>
__device__ __forceinline__ void tmem_load(uint32_t addr, uint32_t* r) {
    if constexpr (N == 16) tmem_ld16(addr, r);
    else {
#pragma unroll
        for (int c = 0; c < N; c += 32) tmem_ld32(addr + c, r + c);
    }
}
// The packed halves (N / 2 values) of N columns.
template <int N>
__device__ __forceinline__ void tmem_store_part(uint32_t addr, const uint32_t* r) {
    if constexpr (N == 32) tmem_st16(addr, r);
    else tmem_st8(addr, r);
}

// ------------------------------------------------------------------------------------------ dQ
// One item of the dQ kernel: 128 query rows of one head, with the key tiles of the three levels that they see.
struct DqItem {
    int b, h, E;                          // E < 0: there is no further item
    int first[3], end[3];
    int m0, m_last;
    DqItem() = default;
    __device__ __forceinline__ DqItem(const BwdTcParams& p, int item) {
        E = -1;
        if (item >= (int)p.dq_items) return;
        const int tiles = p.Tpad / kBlk, bh = item / tiles;
        b = bh / p.H; h = bh - b * p.H;
        m0 = (tiles - 1 - (item - bh * tiles)) * kBlk;          // latest (heaviest) rows of a head first
        m_last = min(m0 + kBlk - 1, p.T - 1);
        E = 0;
#pragma unroll
        for (int l = 0; l < 3; ++l) {
            if (p.n[l] > 0) key_tile_range(l, m0, m_last, p.q_offset, p.window, p.n[l], first[l], end[l]);
            else first[l] = end[l] = 0;
            E += end[l] - first[l];
        }
    }
};

template <int DH>
__global__ void __launch_bounds__(BCfg<DH>::kThreads, 1) bwd_dq_tc_kernel(const __grid_constant__ BwdMaps maps, const BwdTcParams p) {
    using C = BCfg<DH>;
    constexpr uint32_t kColS = 0, kColDP = 256, kColAcc = 384;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    uint8_t* sQ = smem;
    uint8_t* sdO = sQ + C::kTile;
    uint8_t* sK = sdO + C::kTile;                         // kStagesK tiles
    uint8_t* sV = sK + C::kStagesK * C::kTile;            // kStages tiles
    __shared__ BwdBarriers bar;
    __shared__ uint32_t tmem_base_slot;
    __shared__ WaitCtl wait_ctl;
    __shared__ DqItem items[2];
    __shared__ float gsm[C::kGsm][3][kBlk];               // the other warpgroups' sums of a row, on their way to the first

    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // tid >> 5, but provably warp-uniform for the compiler
    if (tid == 0) {
        wait_ctl.abort = 0;
        wait_ctl.limit_ns = p.wait_limit_ns;
        mbar_init(&bar.fixed_full, 1);
        for (int s = 0; s < kMaxStages; ++s) {
            mbar_init(&bar.a_full[s], 1); mbar_init(&bar.a_empty[s], 1);
            mbar_init(&bar.b_full[s], 1); mbar_init(&bar.b_empty[s], 1);
        }
        mbar_init(&bar.s_full[0], 1); mbar_init(&bar.s_full[1], 1);
        mbar_init(&bar.dp_full, 1);
        for (int i = 0; i < 2; ++i) { mbar_init(&bar.p_part[i], C::kEw); mbar_init(&bar.ds_part[i], C::kEw); }   // one arrival per element-wise warp
        mbar_init(&bar.acc_done, 1);
        mbar_init(&bar.fixed_free, 1);
        for (int i = 0; i < 2; ++i) { mbar_init(&bar.item_full[i], 1); mbar_init(&bar.item_free[i], 1 + C::kEw); }   // the issuing warp and the element-wise warps
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // Neither of the two kernels reads what the other writes, so the second one's CTAs start as soon as an SM has no more items of the
    // first, under its tail, instead of at its end.  What the second one reads was there before the first let it start (below); the
    // statistics, which an L1 may still hold from an earlier call, are fetched past it.  Its wait for the first comes at the end: the
    // next kernel waits for the second only and needs both.
    if (p.dq_first) chain_wait();
    else chain_trigger();
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_slot)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (p.dq_first) chain_trigger();                      // only now, with the statistics there for whoever comes next
    const uint32_t tmem = tmem_base_slot;
    volatile WaitCtl* abortp = &wait_ctl;

    if (warp == C::kProducerWarp) {
        int issued_k = 0, issued_v = 0, filled = 0;          // key tiles requested (per ring), items
        bool ok = true;
        // (behind the dK/dV kernel some CTAs start late: all items come from the counter then)
        const int dealt = p.dq_first ? (int)gridDim.x : 0;
        int item = blockIdx.x;
        if (!p.dq_first) {
            if (lane == 0) item = (int)atomicAdd(p.dq_ticket, 1u);
            item = __shfl_sync(0xffffffffu, item, 0);
        }
        for (int it = 0; ok; ++it) {
            const DqItem I(p, item);
            if (!(ok = post_item(bar, items, it, I, lane, abortp)) || I.E < 0) break;
            const int kvh = I.h / p.kv_group;
            if (I.E > 0) {
                // the previous item's Q and dO have had their last reader when its last dP is complete
                if (filled > 0 && !mbar_wait_warp(&bar.fixed_free, (uint32_t)(filled - 1) & 1u, abortp)) { ok = false; break; }
                if (lane == 0) {
                    mbar_expect_tx(&bar.fixed_full, 2 * C::kTile);
#pragma unroll
                    for (int pn = 0; pn < C::kPanels; ++pn) {
                        tma_load_4d(sQ + pn * kPanel, &maps.q, pn * 64, (int)I.m0, I.h, I.b, &bar.fixed_full);
                        tma_load_4d(sdO + pn * kPanel, &maps.dO, pn * 64, (int)I.m0, I.h, I.b, &bar.fixed_full);
                    }
                }
                __syncwarp();
                ++filled;
            }
#pragma unroll 1
            for (int l = 0; l < 3 && ok; ++l) {
                const int kt_end = pick3(I.end, l);
                for (int kt = pick3(I.first, l); kt < kt_end; ++kt) {
                    const int s = issued_k % C::kStagesK, sv = issued_k % C::kStages;
                    const uint32_t ph = (uint32_t)(issued_k / C::kStagesK) & 1u, phv = (uint32_t)(issued_k / C::kStages) & 1u;
                    if (!mbar_wait_warp(&bar.a_empty[s], ph ^ 1u, abortp)) { ok = false; break; }
                    if (lane == 0) {
                        mbar_expect_tx(&bar.a_full[s], C::kTile);
#pragma unroll
                        for (int pn = 0; pn < C::kPanels; ++pn)
                            tma_load_4d(sK + s * C::kTile + pn * kPanel, &maps.k[l], pn * 64, kt * kBlk, kvh, I.b, &bar.a_full[s]);
                    }
                    __syncwarp();
                    ++issued_k;
                    if (!mbar_wait_warp(&bar.b_empty[sv], phv ^ 1u, abortp)) { ok = false; break; }
                    if (lane == 0) {
                        mbar_expect_tx(&bar.b_full[sv], C::kTile);
#pragma unroll
                        for (int pn = 0; pn < C::kPanels; ++pn)
                            tma_load_4d(sV + sv * C::kTile + pn * kPanel, &maps.v[l], pn * 64, kt * kBlk, kvh, I.b, &bar.b_full[sv]);
                    }
                    __syncwarp();
                    ++issued_v;
                }
            }
            // The next item is taken only now, with this one's last tiles still in the rings: taken earlier, the items left
            // for a second round would go to whichever CTAs started first, the ones with the longest items among them.
            if (lane == 0) item = dealt + (int)atomicAdd(p.dq_ticket, 1u);
            item = __shfl_sync(0xffffffffu, item, 0);
        }
        // every copy issued above must have landed before the shared memory can be given up
        const unsigned long long t_drain = gtimer();
        if (filled > 0) mbar_drain(&bar.fixed_full, (uint32_t)(filled - 1) & 1u, abortp, t_drain);
        for (int i = issued_k > C::kStagesK ? issued_k - C::kStagesK : 0; i < issued_k; ++i)
            mbar_drain(&bar.a_full[i % C::kStagesK], (uint32_t)(i / C::kStagesK) & 1u, abortp, t_drain);
        for (int i = issued_v > C::kStages ? issued_v - C::kStages : 0; i < issued_v; ++i)
            mbar_drain(&bar.b_full[i % C::kStages], (uint32_t)(i / C::kStages) & 1u, abortp, t_drain);
    } else if (warp == C::kMmaWarp) {
        {   // every lane runs the issue loop (converged); elect.sync inside the wrappers picks the issuing lane
            // low descriptor words of the operands (see make_desc): K-major views for S and dP, MN-major view of K for dQ
            const uint32_t q_lo = desc_lo_kmajor(smem_u32(sQ)), g_lo = desc_lo_kmajor(smem_u32(sdO));
            const uint32_t k_lo = desc_lo_kmajor(smem_u32(sK)), v_lo = desc_lo_kmajor(smem_u32(sV));
            const uint32_t kt_lo = desc_lo_mnmajor(smem_u32(sK), kPanel);
            // g numbers the CTA's key tiles across its items
            auto issue_s = [&](int g) -> bool {             // S(g) = Q K(g)^T into the ping/pong buffer g & 1
                const int s = g % C::kStagesK;
                if (!mbar_wait_warp(&bar.a_full[s], (uint32_t)(g / C::kStagesK) & 1u, abortp)) return false;
                tc_fence_after();
                const uint32_t ka = k_lo + s * (C::kTile >> 4);
#pragma unroll
                for (int k = 0; k < DH / 16; ++k)
                    mma_ss_elect(tmem + kColS + (g & 1) * 128, make_desc(q_lo + kstep_off(k, kPanel)), make_desc(ka + kstep_off(k, kPanel)),
                           C::kIdescS, k > 0);
                mma_commit_elect(&bar.s_full[g & 1]);
                return true;
            };
            int g = 0, filled = 0;
            bool ok = true;
            for (int it = 0; ok; ++it) {
                DqItem I;
                if (!(ok = take_item(bar, items, it, I, lane, abortp)) || I.E < 0) break;
                const int E = I.E;
                if (E == 0) continue;
                // S(0) and dP(0) of this item run while the element-wise threads still store the previous one's dQ: the
                // accumulator is not touched before those threads hand over the first dS.
                if (!mbar_wait_warp(&bar.fixed_full, (uint32_t)filled & 1u, abortp)) { ok = false; break; }
                ++filled;
                tc_fence_after();
                if (!issue_s(g)) { ok = false; break; }
                for (int e = 0; e < E && ok; ++e, ++g) {
                    const int s = g % C::kStagesK, sv = g % C::kStages;
                    if (!mbar_wait_warp(&bar.b_full[sv], (uint32_t)(g / C::kStages) & 1u, abortp)) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t va = v_lo + sv * (C::kTile >> 4), kta = kt_lo + s * (C::kTile >> 4);
#pragma unroll
                    for (int k = 0; k < DH / 16; ++k)          // dP(e) = dO V(e)^T  (dS(e-1), which shares the columns, was consumed by dQ(e-1) issued before)
                        mma_ss_elect(tmem + kColDP, make_desc(g_lo + kstep_off(k, kPanel)), make_desc(va + kstep_off(k, kPanel)), C::kIdescS, k > 0);
                    mma_commit_elect(&bar.dp_full);
                    mma_commit_elect(&bar.b_empty[sv]);
                    if (e + 1 == E) mma_commit_elect(&bar.fixed_free);
                    if (e + 1 < E && !issue_s(g + 1)) { ok = false; break; }
                    // dQ += dS(e) K(e), in the two parts in which the element-wise threads hand dS over (half of each thread's
                    // columns: at d = 128 K-steps {0, 1, 4, 5}, then {2, 3, 6, 7}), so that the first half runs under the second
#pragma unroll
                    for (int part = 0; part < 2; ++part) {
                        if (!mbar_wait_warp(&bar.ds_part[part], (uint32_t)g & 1u, abortp)) { ok = false; break; }
                        tc_fence_after();
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const int k = C::kstep(part, i);
                            mma_ts_elect(tmem + kColAcc, tmem + kColDP + C::packed_col(k), make_desc(kta + k * (2048 >> 4)), C::kIdescAcc,
                                   (e > 0 || part > 0 || i > 0) ? 1u : 0u);
                        }
                    }
                    if (!ok) break;
                    mma_commit_elect(&bar.a_empty[s]);
                }
                if (ok) mma_commit_elect(&bar.acc_done);
            }
        }
    } else {
        // ------------------------------------------------------------ element-wise warpgroups (thread = query row, 64 of the 128 columns; d = 64: 32)
        const int w = warp >> 2;
        const int r = tid & 127;
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t dp_addr = tmem + lane_base + kColDP + w * C::kCols;
        bool ok = true;
        int g = 0, filled = 0;
#pragma unroll 1
        for (int it = 0;; ++it) {
        // The warps leave together: those that took an item meet at barriers in its epilogue, so none may be missing there.
        DqItem I;
        I.E = -1;
        if (ok) ok = take_item(bar, items, it, I, lane, abortp);
        if (!softmax_group_all<C::kEw>(ok && I.E >= 0)) break;
        const int E = I.E;
        const long long bh = (long long)I.b * p.H + I.h, m0 = I.m0, m_last = I.m_last, t = m0 + r;
        const bool row_valid = t < p.T;
        float Dt = 0.f, bias[3] = {-INFINITY, -INFINITY, -INFINITY};
        if (row_valid) {
            Dt = __ldcg(p.statD + bh * p.Tpad + t);
#pragma unroll
            for (int l = 0; l < 3; ++l) {
                bias[l] = __ldcg(p.statB[l] + bh * p.Tpad + t);
            }
        }
        float Al[3] = {0.f, 0.f, 0.f}, Sl[3] = {0.f, 0.f, 0.f};   // per level: sum p dP and sum p over this thread's columns
#pragma unroll
        for (int l = 0; l < 3; ++l) {
            if (!ok || I.first[l] == I.end[l]) continue;
            long long lo = 0, hi = 0;
            // a row past T has a bias of -inf, so its weights are 0 whatever it sees: it takes the last row's range
            visible_range(l, (row_valid ? t : m_last) + p.q_offset, p.window, p.n[l], 0, lo, hi);
            int full_first = 0, full_end = 0;
            {
                long long lo_f, hi_f, lo_l, hi_l;
                visible_range(l, m0 + p.q_offset, p.window, p.n[l], 0, lo_f, hi_f);
                visible_range(l, m_last + p.q_offset, p.window, p.n[l], 0, lo_l, hi_l);
                full_first = (int)((lo_l + kBlk - 1) / kBlk);
                full_end = (int)(hi_f / kBlk);
            }
            // sums over this thread's columns as packed pairs (even, odd column)
            uint64_t a2 = pack2(0.f, 0.f), z2 = a2;
            const float bl = bias[l];
            const uint64_t scale2 = pack2(p.scale_log2, p.scale_log2), bl2 = pack2(bl, bl), negD2 = pack2(-Dt, -Dt);
            for (int kt = I.first[l]; kt < I.end[l]; ++kt, ++g) {
                // phase 1: p = 2^(s * scale + bias) for this thread's columns (needs S only)
                ok = mbar_wait(&bar.s_full[g & 1], (uint32_t)(g >> 1) & 1u, abortp);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                tc_fence_after();
                float pr[C::kCols];
                tmem_load<C::kCols>(tmem + lane_base + kColS + (g & 1) * 128 + w * C::kCols, reinterpret_cast<uint32_t*>(pr));
                tmem_ld_wait();
                if (!(kt >= full_first && kt < full_end)) {
                    const long long j0 = (long long)kt * kBlk + w * C::kCols;
                    mask_cols(pr, (int)max(0LL, min(lo - j0, (long long)C::kCols)), (int)max(0LL, min(hi - j0, (long long)C::kCols)));
                }
#pragma unroll
                for (int c = 0; c < C::kCols; c += 2) {
                    float x0, x1;
                    unpack2(fma2(pack2(pr[c], pr[c + 1]), scale2, bl2), x0, x1);
                    pr[c] = ex2(x0);
                    pr[c + 1] = ex2(x1);
                    z2 = add2(z2, pack2(pr[c], pr[c + 1]));
                }
                // phase 2: dS = p (dP - D), written (bf16) over the dP columns just read
                ok = mbar_wait(&bar.dp_full, (uint32_t)g & 1u, abortp);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                tc_fence_after();
                float dp[C::kCols];
                tmem_load<C::kCols>(dp_addr, reinterpret_cast<uint32_t*>(dp));
                tmem_ld_wait();
                constexpr int kHalf = C::kCols / 2;
                uint32_t pk[kHalf / 2];
                auto ds_cols = [&](int c_from, int c_to, int c_base) {
#pragma unroll
                    for (int c = c_from; c < c_to; c += 2) {
                        const uint64_t p2 = pack2(pr[c], pr[c + 1]), d2 = pack2(dp[c], dp[c + 1]);
                        a2 = fma2(p2, d2, a2);
                        float s0, s1;
                        unpack2(mul2(p2, add2(d2, negD2)), s0, s1);
                        pk[(c - c_base) / 2] = pack_bf16(s0, s1);
                    }
                };
                auto hand_over = [&](int part) {
                    tmem_st_wait();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&bar.ds_part[part]);
                };
                ds_cols(0, kHalf, 0);
                tmem_store_part<kHalf>(dp_addr, pk);
                ds_cols(kHalf, kHalf + kHalf / 2, kHalf);
                hand_over(0);                                // the first part's store has completed by now
                ds_cols(kHalf + kHalf / 2, C::kCols, kHalf);
                tmem_store_part<kHalf>(dp_addr + kHalf / 2, pk);
                hand_over(1);
            }
            {
                float a0, a1, z0, z1;
                unpack2(a2, a0, a1);
                unpack2(z2, z0, z1);
                Al[l] = a0 + a1;
                Sl[l] = z0 + z1;
            }
        }
        // ------------------------------------------------------------ epilogue
        if (ok && E > 0) {
            ok = mbar_wait(&bar.acc_done, (uint32_t)filled++ & 1u, abortp);
            ok = __all_sync(0xffffffffu, ok);
        }
        if (ok) {
            tc_fence_after();
            const int first_row = (warp & 3) * 32;                     // of this warp, within the tile
            __nv_bfloat16* out = p.dQ + (bh * p.T + m0 + first_row) * DH;
            constexpr int kOut = DH / C::kGroups, kStep = kOut < 32 ? kOut : 32;     // columns of a warpgroup
#pragma unroll
            for (int c0 = w * kOut; c0 < (w + 1) * kOut; c0 += kStep) {
                uint32_t o[kStep];
                if (E > 0) {
                    tmem_load<kStep>(tmem + lane_base + kColAcc + c0, o);
                    tmem_ld_wait();
                } else {
#pragma unroll
                    for (int i = 0; i < kStep; ++i) o[i] = 0u;
                }
                store_rows_bf16<kStep>(out + c0, DH, (int)min(32LL, p.T - m0 - first_row), o, p.scale, lane);
            }
        }
        // Gate-logit gradient of this head: G_l = sum_{j in l} p (dP - D').  D' = sum p dP / sum p equals
        // dO . O in exact arithmetic but does not inherit the rounding of O to bf16, so sum_l G_l = 0 holds
        // to fp32 accuracy.  The two warpgroups hold disjoint columns: add their partial sums first.
        // (A warp that gave up joins these barriers too.)
        float asum[3], zsum[3];
#pragma unroll
        for (int half = 0; half < 2; ++half)
#pragma unroll
            for (int w0 = 1; w0 < C::kGroups; w0 += C::kGsm) {
                if (half || w0 > 1) softmax_group_sync<C::kEw>();
                if (w >= w0 && w < w0 + C::kGsm)
#pragma unroll
                    for (int l = 0; l < 3; ++l) gsm[w - w0][l][r] = half ? Sl[l] : Al[l];
                softmax_group_sync<C::kEw>();
                if (w == 0)
#pragma unroll
                    for (int l = 0; l < 3; ++l) {
                        float v = w0 == 1 ? (half ? Sl[l] : Al[l]) : (half ? zsum[l] : asum[l]);
#pragma unroll
                        for (int i = 0; i < C::kGsm; ++i) v += gsm[i][l][r];
                        (half ? zsum : asum)[l] = v;
                    }
            }
        if (w == 0 && ok && row_valid) {
            const float ztot = zsum[0] + zsum[1] + zsum[2];
            const float dd = ztot > 0.f ? (asum[0] + asum[1] + asum[2]) / ztot : 0.f;
            float* gp = p.Gpart + (bh * p.T + t) * 3;
#pragma unroll
            for (int l = 0; l < 3; ++l) gp[l] = asum[l] - zsum[l] * dd;
        }
        }   // items
    }

    tc_fence_before();
    __syncthreads();
    if (tid == 0 && wait_ctl.abort) atomicExch(p.status, (unsigned int)MKA_ERR_TIMEOUT);
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
    chain_wait();
}

// ------------------------------------------------------------------------------------------ dK, dV
// One item of the dK/dV kernel: a key tile of one level and KV head, with the query tiles that see it.
struct DkvItem {
    int b, h, lvl, first, Eq, E;          // h: KV head; its query heads are h * G .. h * G + G - 1;  E < 0: there is no further item
    int n, j0, j_last;                    // (levels of this path hold fewer than 2^31 - 256 rows)
    DkvItem() = default;
    __device__ __forceinline__ DkvItem(const BwdTcParams& p, int item) {
        E = -1;
        if (item >= (int)p.dkv_items) return;
        const int tiles = p.kv_tiles[0] + p.kv_tiles[1] + p.kv_tiles[2], bh = item / tiles;
        int kt = item - bh * tiles;
        b = bh / p.H_kv; h = bh - b * p.H_kv;
        // key tiles of a head in decreasing order of work: L3 (seen by every query), L2 from the oldest key on, L1
        lvl = 2;
        if (kt >= p.kv_tiles[2]) { kt -= p.kv_tiles[2]; lvl = 1; if (kt >= p.kv_tiles[1]) { kt -= p.kv_tiles[1]; lvl = 0; } }
        n = (int)pick3(p.n, lvl);
        j0 = kt * kBlk;
        j_last = min(j0 + kBlk - 1, n - 1);
        // queries t (position t + q_offset) that can see a key of this tile
        long long t_lo = 0, t_hi = p.T;
        if (lvl == 0) { t_lo = (long long)j0 - p.q_offset; t_hi = (long long)j_last + p.window - p.q_offset; }
        else if (lvl == 1) { t_lo = (long long)j0 - p.q_offset; }
        if (t_lo < 0) t_lo = 0;
        if (t_hi > p.T) t_hi = p.T;
        first = t_hi > t_lo ? (int)(t_lo / kBlk) : 0;
        Eq = t_hi > t_lo ? (int)((t_hi + kBlk - 1) / kBlk) - first : 0;    // query tiles of ONE head that see this key tile
        E = Eq * p.kv_group;                                                // the stream: head by head, each head's tiles in order
    }
};

template <int DH>
__global__ void __launch_bounds__(BCfg<DH>::kThreadsDkv, 1) bwd_dkv_tc_kernel(const __grid_constant__ BwdMaps maps, const BwdTcParams p) {
    using C = BCfg<DH>;
    constexpr uint32_t kColS = 0, kColDP = 128, kColDK = 256, kColDV = 256 + DH;
    // d = 64 leaves room for a second S^T: S^T(g+1) is multiplied while the element-wise threads still work on S^T(g).
    constexpr bool kTwoS = DH == 64;
    constexpr uint32_t kColS1 = kTwoS ? 384 : kColS;
    static_assert(!kTwoS || kColDV + DH <= kColS1, "TMEM columns exceeded");
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    uint8_t* sK = smem;
    uint8_t* sV = sK + C::kTile;
    uint8_t* sQ = sV + C::kTile;                          // kStages tiles
    uint8_t* sdO = sQ + C::kStages * C::kTile;            // kStages tiles
    // Operand slabs of the extra K-step (16 columns, no swizzle: 8-row x 16-byte core matrices, the two of a row group
    // 128 bytes apart, row groups 256 bytes apart).  sAugQ: per stage, [query][k] = the query's exponent bias divided by
    // the score scale, split into three bf16 terms (k = 0..2), then [query][k] = -D_t split the same way; sAugK: ones in
    // k = 0..2 for every key.  S^T + bias / scale and dP^T - D then come out of the tensor pipe, and the element-wise
    // threads need no per-column operand at all.
    uint8_t* sAugQ = sdO + C::kStages * C::kTile;          // kStages x {bias slab, D slab}
    uint8_t* sAugK = sAugQ + C::kStages * 2 * C::kAugBytes;
    __shared__ BwdBarriers bar;
    __shared__ uint32_t tmem_base_slot;
    __shared__ WaitCtl wait_ctl;
    __shared__ DkvItem items[2];
    __shared__ unsigned int gate_chunk;

    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // tid >> 5, but provably warp-uniform for the compiler
    if (warp == C::kProducerWarp && lane == 0) {
        wait_ctl.abort = 0;
        wait_ctl.limit_ns = p.wait_limit_ns;
        mbar_init(&bar.fixed_full, 1);
        for (int s = 0; s < kMaxStages; ++s) {               // full: the copy's bytes and the slab
            mbar_init(&bar.a_full[s], 2); mbar_init(&bar.a_empty[s], 1);
            mbar_init(&bar.b_full[s], 2); mbar_init(&bar.b_empty[s], 1);
        }
        mbar_init(&bar.s_full[0], 1); mbar_init(&bar.s_full[1], 1);
        mbar_init(&bar.dp_full, 1);
        for (int i = 0; i < 2; ++i) { mbar_init(&bar.p_part[i], C::kEw); mbar_init(&bar.ds_part[i], C::kEw); }   // one arrival per element-wise warp
        mbar_init(&bar.acc_done, 1);
        mbar_init(&bar.fixed_free, 1);
        for (int i = 0; i < 2; ++i) { mbar_init(&bar.item_full[i], 1); mbar_init(&bar.item_free[i], 3 + C::kEw); }   // the issuing, the slab and the element-wise warps
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // every slab zero (columns 3..15 stay zero), ones for the keys: all threads share the 36 KB
    for (int i = tid; i < (int)((C::kStages * 2 + 1) * C::kAugBytes / 16); i += C::kThreadsDkv)
        reinterpret_cast<uint4*>(sAugQ)[i] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    if (tid < kBlk) *reinterpret_cast<uint4*>(sAugK + (tid & 7) * 16 + (tid >> 3) * 256) = make_uint4(0x3f803f80u, 0x00003f80u, 0u, 0u);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    // (see the dQ kernel; written over keys or values that the dQ kernel reads, dK and dV wait for its end)
    const bool waits = !p.dq_first || p.in_place;
    if (waits) chain_wait();
    else chain_trigger();
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_slot)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (waits) chain_trigger();
    const uint32_t tmem = tmem_base_slot;
    volatile WaitCtl* abortp = &wait_ctl;

    if (warp == C::kProducerWarp) {
        int issued = 0, issued_b = 0, filled = 0;            // query tiles requested (per ring), items with tiles
        bool ok = true;
        int item = blockIdx.x;
        for (int it = 0; ok; ++it) {
            const DkvItem I(p, item);
            if (!(ok = post_item(bar, items, it, I, lane, abortp)) || I.E < 0) break;
            if (I.E > 0) {
                // the previous item's K and V have had their last reader when its last dP^T is complete
                if (filled > 0 && !mbar_wait_warp(&bar.fixed_free, (uint32_t)(filled - 1) & 1u, abortp)) { ok = false; break; }
                if (lane == 0) {
                    mbar_expect_tx(&bar.fixed_full, 2 * C::kTile);
#pragma unroll
                    for (int pn = 0; pn < C::kPanels; ++pn) {
                        tma_load_4d(sK + pn * kPanel, &maps.k[I.lvl], pn * 64, (int)I.j0, I.h, I.b, &bar.fixed_full);
                        tma_load_4d(sV + pn * kPanel, &maps.v[I.lvl], pn * 64, (int)I.j0, I.h, I.b, &bar.fixed_full);
                    }
                }
                __syncwarp();
                ++filled;
                int hq = I.h * p.kv_group, eq = 0;           // query head and tile-within-head of tile e
                // Two rings: a stage's dO tile is free again after dV of its tile, its Q tile only after dK, one product later;
                // and the next tile's Q is what the issuing warp waits for first.  Each is re-filled as soon as it is free.
                for (int e = 0; e < I.E; ++e) {
                    const int s = issued % C::kStages;
                    const uint32_t ph = (uint32_t)(issued / C::kStages) & 1u;
                    if (p.test_stall && e == I.E - 1) { ok = false; break; }       // test hook: the last tile never arrives
                    const int tt = (I.first + eq) * kBlk;
                    if (!mbar_wait_warp(&bar.b_empty[s], ph ^ 1u, abortp)) { ok = false; break; }
                    if (lane == 0) {
                        mbar_expect_tx(&bar.b_full[s], C::kTile);
#pragma unroll
                        for (int pn = 0; pn < C::kPanels; ++pn)
                            tma_load_4d(sdO + s * C::kTile + pn * kPanel, &maps.dO, pn * 64, tt, hq, I.b, &bar.b_full[s]);
                    }
                    __syncwarp();
                    ++issued_b;
                    if (!mbar_wait_warp(&bar.a_empty[s], ph ^ 1u, abortp)) { ok = false; break; }
                    if (lane == 0) {
                        mbar_expect_tx(&bar.a_full[s], C::kTile);
#pragma unroll
                        for (int pn = 0; pn < C::kPanels; ++pn)
                            tma_load_4d(sQ + s * C::kTile + pn * kPanel, &maps.q, pn * 64, tt, hq, I.b, &bar.a_full[s]);
                    }
                    __syncwarp();
                    ++issued;
                    if (++eq == I.Eq) { eq = 0; ++hq; }
                }
            }
            // The next item is taken only now, with this one's last tiles still in the rings: taken earlier, the items left
            // for a second round would go to whichever CTAs started first, the ones with the longest items among them.
            if (lane == 0) item = (int)gridDim.x + (int)atomicAdd(p.dkv_ticket, 1u);
            item = __shfl_sync(0xffffffffu, item, 0);
        }
        // every copy issued above must have landed before the shared memory can be given up (a stage that a slab warp gave up
        // before writing does not complete: the limit, one for all of these waits, ends it)
        const unsigned long long t_drain = gtimer();
        if (filled > 0) mbar_drain(&bar.fixed_full, (uint32_t)(filled - 1) & 1u, abortp, t_drain);
        for (int i = issued > C::kStages ? issued - C::kStages : 0; i < issued; ++i)
            mbar_drain(&bar.a_full[i % C::kStages], (uint32_t)(i / C::kStages) & 1u, abortp, t_drain);
        for (int i = issued_b > C::kStages ? issued_b - C::kStages : 0; i < issued_b; ++i)
            mbar_drain(&bar.b_full[i % C::kStages], (uint32_t)(i / C::kStages) & 1u, abortp, t_drain);
        if (lane == 0) gate_chunk = atomicAdd(p.gate_ticket, 1u);
    } else if (warp == C::kSlabWarp || warp == C::kSlabWarp + 1) {
        // The operand slabs of the ninth K-step: the first of these warps writes the bias slabs (ring of the Q tiles), the second
        // the D slabs (ring of the dO tiles), four queries a lane, fetched one tile ahead.  Warps of their own: when the
        // warp that issues the copies wrote them too, its loop took 2400 cycles a tile and everything waited for it.
        const bool is_d = warp != C::kSlabWarp;
        uint64_t *const full = is_d ? bar.b_full : bar.a_full, *const empty = is_d ? bar.b_empty : bar.a_empty;
        uint8_t* const slab = sAugQ + (is_d ? C::kAugBytes : 0);
        const float mul = is_d ? -1.f : 1.f / p.scale_log2;
        int n_out = 0;
        bool ok = true;
        for (int it = 0; ok; ++it) {
            DkvItem I;
            if (!(ok = take_item(bar, items, it, I, lane, abortp)) || I.E < 0) break;
            const float* src = (is_d ? p.statD : pick3(p.statB, I.lvl)) + ((long long)I.b * p.H + (long long)I.h * p.kv_group) * p.Tpad +
                               (long long)I.first * kBlk + 4 * lane;
            int eq = 0;
            float4 next = make_float4(0.f, 0.f, 0.f, 0.f);
            if (I.E > 0) next = __ldcg(reinterpret_cast<const float4*>(src));
            for (int e = 0; e < I.E; ++e, ++n_out) {
                const int s = n_out % C::kStages;
                const float v[4] = {next.x * mul, next.y * mul, next.z * mul, next.w * mul};
                if (++eq == I.Eq) { eq = 0; src += p.Tpad; }
                if (e + 1 < I.E) next = __ldcg(reinterpret_cast<const float4*>(src + (long long)eq * kBlk));
                uint4 row[4];                                        // each value as three bf16 terms
#pragma unroll
                for (int i = 0; i < 4; ++i) row[i] = split3_bf16(v[i]);
                if (!mbar_wait_warp(&empty[s], ((uint32_t)(n_out / C::kStages) & 1u) ^ 1u, abortp)) { ok = false; break; }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int r = 4 * lane + i;
                    *reinterpret_cast<uint4*>(slab + s * 2 * C::kAugBytes + (r & 7) * 16 + (r >> 3) * 256) = row[i];
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(&full[s]);
            }
        }
    } else if (warp == C::kMmaWarp) {
        {   // every lane runs the issue loop (converged); elect.sync inside the wrappers picks the issuing lane
            // low descriptor words (see make_desc): K-major views for S^T and dP^T, MN-major views of Q and dO for dK and dV
            const uint32_t k_lo = desc_lo_kmajor(smem_u32(sK)), v_lo = desc_lo_kmajor(smem_u32(sV));
            const uint32_t q_lo = desc_lo_kmajor(smem_u32(sQ)), g_lo = desc_lo_kmajor(smem_u32(sdO));
            const uint32_t qt_lo = desc_lo_mnmajor(smem_u32(sQ), kPanel), gt_lo = desc_lo_mnmajor(smem_u32(sdO), kPanel);
            const uint32_t augk_lo = desc_lo_flat(smem_u32(sAugK)), augq_lo = desc_lo_flat(smem_u32(sAugQ));
            // g numbers the CTA's query tiles across its items
            auto issue_s = [&](int g) {                     // S^T(g) = K Q(g)^T   (P^T(g-1), which shares the columns, was consumed by dV(g-1) issued before; Q(g) has landed)
                const int s = g % C::kStages;
                tc_fence_after();
                const uint32_t qa = q_lo + s * (C::kTile >> 4);
                const uint32_t s_col = (g & 1) ? kColS1 : kColS;
#pragma unroll
                for (int k = 0; k < DH / 16; ++k)
                    mma_ss_elect(tmem + s_col, make_desc(k_lo + kstep_off(k, kPanel)), make_desc(qa + kstep_off(k, kPanel)), C::kIdescS, k > 0);
                mma_ss_elect(tmem + s_col, make_desc_flat(augk_lo), make_desc_flat(augq_lo + s * (2 * C::kAugBytes >> 4)), C::kIdescS, 1u);   // + bias_t / scale
                mma_commit_elect(&bar.s_full[kTwoS ? g & 1 : 0]);
            };
            auto issue_dp = [&](int g) -> bool {            // dP^T(g) = V dO(g)^T
                if (!mbar_wait_warp(&bar.b_full[g % C::kStages], (uint32_t)(g / C::kStages) & 1u, abortp)) return false;
                tc_fence_after();
                const uint32_t ga = g_lo + (g % C::kStages) * (C::kTile >> 4);
#pragma unroll
                for (int k = 0; k < DH / 16; ++k)
                    mma_ss_elect(tmem + kColDP, make_desc(v_lo + kstep_off(k, kPanel)), make_desc(ga + kstep_off(k, kPanel)), C::kIdescS, k > 0);
                mma_ss_elect(tmem + kColDP, make_desc_flat(augk_lo), make_desc_flat(augq_lo + ((g % C::kStages) * 2 + 1) * (C::kAugBytes >> 4)), C::kIdescS, 1u);   // - D_t
                mma_commit_elect(&bar.dp_full);
                return true;
            };
            int g = 0, filled = 0;
            bool ok = true;
            for (int it = 0; ok; ++it) {
                DkvItem I;
                if (!(ok = take_item(bar, items, it, I, lane, abortp)) || I.E < 0) break;
                const int E = I.E;
                if (E == 0) continue;
                // S^T(0) and dP^T(0) of this item run while the element-wise threads still store the previous one's dK and
                // dV: the accumulators are not touched before those threads hand over the first P^T.
                if (!mbar_wait_warp(&bar.fixed_full, (uint32_t)filled & 1u, abortp) ||
                    !mbar_wait_warp(&bar.a_full[g % C::kStages], (uint32_t)(g / C::kStages) & 1u, abortp)) { ok = false; break; }
                ++filled;
                issue_s(g);
                if (!issue_dp(g)) { ok = false; break; }
                if (E == 1) mma_commit_elect(&bar.fixed_free);
                auto wait_q = [&](int gq) { return mbar_wait_warp(&bar.a_full[gq % C::kStages], (uint32_t)(gq / C::kStages) & 1u, abortp); };
                if (kTwoS && E > 1) {
                    if (!wait_q(g + 1)) { ok = false; break; }
                    issue_s(g + 1);
                }
                for (int e = 0; e < E && ok; ++e, ++g) {
                    const uint32_t s_col = (g & 1) ? kColS1 : kColS;
                    const int s = g % C::kStages;
                    const uint32_t qta = qt_lo + s * (C::kTile >> 4), gta = gt_lo + s * (C::kTile >> 4);
                    // dV += P^T(e) dO(e) and dK += dS^T(e) Q(e), each in the two parts in which the element-wise threads
                    // hand their columns over (d = 128: K-steps {0, 1, 4, 5}, then {2, 3, 6, 7}; d = 64: the whole tile at once for dV)
#pragma unroll
                    for (int part = 0; part < 2; ++part) {
                        // (with two S^T the element-wise threads are ahead: one wait, for the whole tile, costs less than two)
                        if (!kTwoS || part == 0) {
                            if (!mbar_wait_warp(&bar.p_part[kTwoS ? g & 1 : part], (uint32_t)(kTwoS ? g >> 1 : g) & 1u, abortp)) { ok = false; break; }
                            tc_fence_after();
                        }
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const int k = C::kstep(part, i);
                            mma_ts_elect(tmem + kColDV, tmem + s_col + C::packed_col(k), make_desc(gta + k * (2048 >> 4)), C::kIdescAcc,
                                   (e > 0 || part > 0 || i > 0) ? 1u : 0u);
                        }
                    }
                    if (!ok) break;
                    mma_commit_elect(&bar.b_empty[s]);                     // dO(e) has had its last reader
                    // S^T(g+1) needs Q(g+1), which can only be requested once dK(g-1) has released its stage; dK(g) needs dS^T(g)
                    // from the element-wise threads.  Either may be ready first, and neither may wait for the other (a late
                    // dK delays the release, the release the copy, the copy the next S^T): whichever comes first goes out first.
                    // The polls stand apart from the products: inside a polling loop the operands of a product are moved
                    // to uniform registers one by one, and the four products of a part took 390 cycles to issue
                    // instead of 36.
                    const uint32_t phg = (uint32_t)g & 1u;
                    uint64_t* const q_bar = &bar.a_full[(g + 1) % C::kStages];
                    const uint32_t q_ph = (uint32_t)((g + 1) / C::kStages) & 1u;
                    auto issue_dk = [&](int part) {
                        tc_fence_after();
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const int k = C::kstep(part, i);
                            mma_ts_elect(tmem + kColDK, tmem + kColDP + C::packed_col(k), make_desc(qta + k * (2048 >> 4)), C::kIdescAcc,
                                         (e > 0 || part > 0 || i > 0) ? 1u : 0u);
                        }
                    };
                    if constexpr (kTwoS) {
                        // S^T(g+1) is long there; behind dK(g) follow dP^T(g+1) and S^T(g+2), whose columns dV(g) has read
                        if (!mbar_wait_warp(&bar.ds_part[1], phg, abortp)) { ok = false; break; }
                        issue_dk(0);
                        issue_dk(1);
                        mma_commit_elect(&bar.a_empty[s]);
                        if (e + 1 < E) {
                            if (!issue_dp(g + 1)) { ok = false; break; }
                            if (e + 2 == E) mma_commit_elect(&bar.fixed_free);
                        }
                        if (e + 2 < E) {
                            if (!wait_q(g + 2)) { ok = false; break; }
                            issue_s(g + 2);
                        }
                        continue;
                    }
                    if (e + 1 < E) {
                        const int first = poll_two(q_bar, q_ph, &bar.ds_part[0], phg, abortp);
                        if (first < 0) { ok = false; break; }
                        if (first == 0) {
                            issue_s(g + 1);
                            if (!mbar_wait_warp(&bar.ds_part[0], phg, abortp)) { ok = false; break; }
                            issue_dk(0);
                            if (!mbar_wait_warp(&bar.ds_part[1], phg, abortp)) { ok = false; break; }
                            issue_dk(1);
                        } else {
                            issue_dk(0);
                            const int second = poll_two(q_bar, q_ph, &bar.ds_part[1], phg, abortp);
                            if (second < 0) { ok = false; break; }
                            if (second == 0) {
                                issue_s(g + 1);
                                if (!mbar_wait_warp(&bar.ds_part[1], phg, abortp)) { ok = false; break; }
                                issue_dk(1);
                            } else {
                                issue_dk(1);
                                if (!mbar_wait_warp(q_bar, q_ph, abortp)) { ok = false; break; }
                                issue_s(g + 1);
                            }
                        }
                    } else {
                        if (!mbar_wait_warp(&bar.ds_part[0], phg, abortp)) { ok = false; break; }
                        issue_dk(0);
                        if (!mbar_wait_warp(&bar.ds_part[1], phg, abortp)) { ok = false; break; }
                        issue_dk(1);
                    }
                    mma_commit_elect(&bar.a_empty[s]);
                    if (e + 1 < E) {
                        if (!issue_dp(g + 1)) { ok = false; break; }
                        if (e + 2 == E) mma_commit_elect(&bar.fixed_free);
                    }
                }
                if (ok) mma_commit_elect(&bar.acc_done);
            }
        }
    } else {
        // ------------------------------------------------------------ element-wise warpgroups (thread = key row, 64 of the 128 query columns; d = 64: 32)
        const int w = warp >> 2;
        const int r = tid & 127;
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t dp_addr = tmem + lane_base + kColDP + w * C::kCols;
        bool ok = true;
        int g = 0, filled = 0;
#pragma unroll 1
        for (int it = 0; ok; ++it) {
        DkvItem I;
        if (!(ok = take_item(bar, items, it, I, lane, abortp)) || I.E < 0) break;
        const int lvl = I.lvl, E = I.E, Eq = I.Eq, first = I.first;
        const long long j0 = I.j0, j_last = I.j_last, j = j0 + r;
        const bool row_valid = j < I.n;
        // queries [q_lo, q_hi) that see key j (the bound t < T is carried by the padded biases)
        // a key past n has its own row of dK and dV, which nobody stores: it takes the last key's range and needs no mask
        const long long j_see = row_valid ? j : j_last;
        const long long q_lo = lvl == 2 ? 0 : j_see - p.q_offset;
        const long long q_hi = lvl == 0 ? j_see + p.window - p.q_offset : (long long)p.Tpad;
        int eq = 0;                                                    // tile within the current query head
        for (int e = 0; e < E; ++e, ++g) {
            const long long tt = (long long)(first + eq) * kBlk;       // first query of the tile
            if (++eq == Eq) eq = 0;
            // phase 1: P^T = 2^(scale * (s + bias_t / scale)) for this thread's query columns; the sum comes from the tensor pipe
            ok = kTwoS ? mbar_wait(&bar.s_full[g & 1], (uint32_t)(g >> 1) & 1u, abortp) : mbar_wait(&bar.s_full[0], (uint32_t)g & 1u, abortp);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc_fence_after();
            const uint32_t s_addr = tmem + lane_base + ((g & 1) ? kColS1 : kColS) + w * C::kCols;
            float pr[C::kCols];
            tmem_load<C::kCols>(s_addr, reinterpret_cast<uint32_t*>(pr));
            tmem_ld_wait();
            // tiles whose every (key, query) pair is visible need no mask
            bool full = true;
            if (lvl != 2) full = full && (j_last - p.q_offset <= tt);
            if (lvl == 0) full = full && (j0 + p.window - p.q_offset >= tt + kBlk);
            if (!full) {
                const long long c0 = tt + w * C::kCols;
                mask_cols(pr, (int)max(0LL, min(q_lo - c0, (long long)C::kCols)), (int)max(0LL, min(q_hi - c0, (long long)C::kCols)));
            }
            constexpr int kHalf = C::kCols / 2;
            // P^T rounded to bf16 for dV.  Phase 2 takes the weights as they are, from pr: widened from here again they cost a quarter of its
            // and phase 1's instructions (backward of [8, 16, 2048, 64] 786 -> 780 us, [2, 16 on 4, 1000, 128] 94.6 -> 93.8).
            uint32_t pk[kHalf];
            const uint64_t scale2 = pack2(p.scale_log2, p.scale_log2);
            auto p_cols = [&](int c_from, int c_to) {
#pragma unroll
                for (int c = c_from; c < c_to; c += 2) {
                    float x0, x1;
                    unpack2(mul2(pack2(pr[c], pr[c + 1]), scale2), x0, x1);
                    // d = 128: every fourth pair on the FMA pipe: the hand-over of P^T, not these threads' total work, is what the
                    // next score product waits for, and the special-function unit alone is the slower way there.  With two S^T it is not
                    // waited for, and the sixteen warps are short of issue slots (65 % used, the special-function unit 25 %, with every
                    // other pair on the FMA pipe).  Backward, us, every other / third / fourth / no pair: [4, 16, 8192, 128] 5622 / 5560 / [5564] / 5709,
                    // [2, 16 on 4, 1000, 128] 96.1 / 94.6 / [95.0] / 95.6; [8, 16, 2048, 64] 803 / - / 791 / [786].
                    float p0, p1;
                    if (kTwoS || (c >> 1) % 4 != 0) { p0 = ex2(x0); p1 = ex2(x1); }
                    else exp2_pair_fma(x0, x1, p0, p1);
                    pk[c / 2] = pack_bf16(p0, p1);
                    pr[c] = p0; pr[c + 1] = p1;
                }
            };
            auto hand_over = [&](uint64_t* bar_part) {       // everything stored so far is in TMEM
                tmem_st_wait();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_part);
            };
            // each half of the thread's columns goes out as soon as it is ready; the first half is handed over in
            // the middle of the second half's exponentials, when its store has long completed
            p_cols(0, kHalf);
            tmem_store_part<kHalf>(s_addr, pk);
            p_cols(kHalf, kHalf + kHalf / 2);
            if constexpr (!kTwoS) hand_over(&bar.p_part[0]);
            p_cols(kHalf + kHalf / 2, C::kCols);
            tmem_store_part<kHalf>(s_addr + kHalf / 2, pk + kHalf / 2);
            // With two S^T a warp may reach this line for tile g+1 while another has not yet for tile g (S^T(g+1) waits for nobody
            // here), and an mbarrier counts arrivals, not warps: each buffer has a barrier of its own.  S^T(g+2) is issued behind
            // dV(g), so no warp arrives twice in one phase.
            hand_over(&bar.p_part[kTwoS ? g & 1 : 1]);
            // phase 2: dS^T = P^T (dP^T - D_t), written over the columns just read; the difference comes from the tensor pipe
            ok = mbar_wait(&bar.dp_full, (uint32_t)g & 1u, abortp);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc_fence_after();
            float dp[C::kCols];
            tmem_load<C::kCols>(dp_addr, reinterpret_cast<uint32_t*>(dp));
            tmem_ld_wait();
            auto ds_cols = [&](int c_from, int c_to) {
#pragma unroll
                for (int c = c_from; c < c_to; c += 2) {
                    float s0, s1;
                    unpack2(mul2(pack2(pr[c], pr[c + 1]), pack2(dp[c], dp[c + 1])), s0, s1);   // p (dP - D)
                    pk[c / 2] = pack_bf16(s0, s1);
                }
            };
            ds_cols(0, kHalf);
            tmem_store_part<kHalf>(dp_addr, pk);
            ds_cols(kHalf, kHalf + kHalf / 2);
            hand_over(&bar.ds_part[0]);
            ds_cols(kHalf + kHalf / 2, C::kCols);
            tmem_store_part<kHalf>(dp_addr + kHalf / 2, pk + kHalf / 2);
            hand_over(&bar.ds_part[1]);
        }
        // ------------------------------------------------------------ epilogue
        if (ok && E > 0) {
            ok = mbar_wait(&bar.acc_done, (uint32_t)filled++ & 1u, abortp);
            ok = __all_sync(0xffffffffu, ok);
        }
        if (ok) {
            tc_fence_after();
            // half of the warpgroups write dK, the others dV, each its share of the columns
            const bool is_k = w < C::kGroups / 2;
            constexpr int kOut = 2 * DH / C::kGroups;
            const int c_first = (is_k ? w : w - C::kGroups / 2) * kOut;
            const int first_row = (warp & 3) * 32;                     // of this warp, within the tile
            const LevelGradDev dL = p.dL[lvl];
            __nv_bfloat16* out = static_cast<__nv_bfloat16*>(is_k ? dL.dk : dL.dv) + I.b * dL.sb + I.h * dL.sh + (j0 + first_row) * dL.sn;
            const float mul = is_k ? p.scale : 1.f;
#pragma unroll
            for (int c0 = c_first; c0 < c_first + kOut; c0 += 32) {
                uint32_t o[32];
                if (E > 0) {
                    tmem_ld32(tmem + lane_base + (is_k ? kColDK : kColDV) + c0, o);
                    tmem_ld_wait();
                } else {
#pragma unroll
                    for (int i = 0; i < 32; ++i) o[i] = 0u;
                }
                store_rows_bf16<32>(out + c0, dL.sn, (int)min(32LL, (long long)I.n - j0 - first_row), o, mul, lane);
            }
        }
        }   // items
    }

    tc_fence_before();
    __syncthreads();
    if (tid == 0 && wait_ctl.abort) atomicExch(p.status, (unsigned int)MKA_ERR_TIMEOUT);
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
    // The gate gradient's sums over the heads, left to the CTAs that are done with their key tiles first: a ticket is a sum per
    // thread, the first one taken under the epilogue.  As a launch behind this one they took 5 us: a step at [1, 8, 700, 128] 60.0 -> 57.6.
    chain_wait();
    const long long per_batch = p.T * 3LL;
    for (;;) {
        const long long at = (long long)gate_chunk * C::kThreadsDkv + tid;
        if (!p.dG || at - tid >= per_batch * p.B) break;
        if (at < per_batch * p.B) sum_dgate(p.Gpart, p.dG, p.H, p.T, at / per_batch, at % per_batch);
        __syncthreads();
        if (tid == 0) gate_chunk = atomicAdd(p.gate_ticket, 1u);
        __syncthreads();
    }
}

template <int DH>
cudaError_t launch_t(const BwdParams& bp, unsigned int* status_word, cudaStream_t st) {
    using C = BCfg<DH>;
    const int Tpad = (bp.T + kBlk - 1) / kBlk * kBlk;
    const long long rows_pad = (long long)bp.B * bp.H * Tpad;
    float* statD = bp.stats;                              // the workspace holds D and the three bias arrays back to back
    float* statB[3];
    for (int l = 0; l < 3; ++l) statB[l] = bp.stats + (long long)(1 + l) * rows_pad;
    const long long sq_n = DH, sq_h = (long long)bp.T * DH, sq_b = (long long)bp.H * bp.T * DH;

    constexpr int kPrepRowsPerBlock = 8 * (32 / (DH / 8)) * 4;          // 8 warps x rows per pass x passes
    cudaError_t e = launch_chained(bwd_prep_kernel<DH>, dim3((Tpad + kPrepRowsPerBlock - 1) / kPrepRowsPerBlock, bp.H, bp.B), dim3(256), 0, st, 0,
                                   static_cast<const __nv_bfloat16*>(bp.O), static_cast<const __nv_bfloat16*>(bp.dO), bp.LSE, bp.gate, bp.H, bp.T,
                                   Tpad, statD, statB[0], statB[1], statB[2], status_word);
    if (e != cudaSuccess) return e;

    BwdTcParams p;
    p.dQ = static_cast<__nv_bfloat16*>(bp.dQ);
    p.statD = statD;
    p.Gpart = bp.Gpart;
    for (int l = 0; l < 3; ++l) {
        p.statB[l] = statB[l];
        p.dL[l] = bp.dL[l];
        p.n[l] = bp.L[l].n;
        p.kv_tiles[l] = (int)((bp.L[l].n + 127) / 128);
    }
    p.B = bp.B; p.H = bp.H; p.T = bp.T; p.Tpad = Tpad; p.kv_group = bp.kv_group > 0 ? bp.kv_group : 1;
    const int H_kv = p.H_kv = bp.H / p.kv_group;
    p.window = bp.window; p.q_offset = bp.q_offset;
    p.scale = bp.scale; p.scale_log2 = bp.scale * kLog2e;
    p.status = status_word;
    p.wait_limit_ns = wait_limit_ns();
    p.test_stall = bp.test_stall;

    // both kernels move 128-row tiles (box = 64 columns x 128 rows)
    BwdMaps m;
    if (!make_bf16_map(&m.q, bp.Q, DH, bp.T, bp.H, bp.B, sq_n, sq_h, sq_b, kBlk) ||
        !make_bf16_map(&m.dO, bp.dO, DH, bp.T, bp.H, bp.B, sq_n, sq_h, sq_b, kBlk))
        return cudaErrorNotSupported;
    for (int l = 0; l < 3; ++l) {
        if (bp.L[l].n == 0) { m.k[l] = m.q; m.v[l] = m.q; continue; }
        if (!make_bf16_map(&m.k[l], bp.L[l].k, DH, bp.L[l].n, H_kv, bp.B, bp.L[l].sn, bp.L[l].sh, bp.L[l].sb, kBlk) ||
            !make_bf16_map(&m.v[l], bp.L[l].v, DH, bp.L[l].n, H_kv, bp.B, bp.L[l].sn, bp.L[l].sh, bp.L[l].sb, kBlk))
            return cudaErrorNotSupported;
    }
    p.dq_items = (long long)(Tpad / kBlk) * bp.H * bp.B;
    p.dq_ticket = status_word + 2;
    p.dkv_items = (long long)(p.kv_tiles[0] + p.kv_tiles[1] + p.kv_tiles[2]) * H_kv * bp.B;
    p.dkv_ticket = status_word + 1;
    p.gate_ticket = status_word + 3;
    p.in_place = bp.in_place;
    // Which of the two comes first: the one with the longer items, which would leave a tail behind the other; the shorter ones then fill the SMs
    // beside them.  An item of dK/dV walks up to every query tile of a group of heads, one of dQ the key tiles of three levels.  dK and dV
    // have to be worth it: the gate gradient's sums, which need all of dQ, are a launch of their own behind it.  Nothing is to be gained with few
    // query tiles or where all items find an SM of their own.  With one or two heads of many tiles dQ's items all start at once,
    // and the SMs with the longest of them would come last to dK/dV's first.  Longest items in tiles (dK/dV, dQ); us of a backward, dQ first /
    // dK and dV first, the pick in brackets:
    //   grouped     [2, 12 on 4, 1100, 64] (27, 13) 86 / [78]        [2, 16 on 4, 1000, 128] (32, 16) 141 / [131]     [1, 16 on 4, 700, 128] (24, 22) 99 / [93]
    //               [1, 28 on 4, 2000, 128] (112, 21) 294 / [248]    [2, 32 on 8, 4096, 128] (128, 46) 1500 / [1414]  [2, 16 on 8, 1600, 128] (26, 19) 153 / [146]
    //               [4, 16 on 8, 2048, 64] (32, 30) [354] / 358      [1, 4 on 2, 2048, 128] (32, 24), 136 items [66] / 68
    //   ungrouped   [1, 8, 3100, 128] (25, 39) [151] / 159           [1, 3, 6000, 64] (47, 61) [116] / 126            [2, 16, 3100, 64] (25, 39) [332] / 342
    //               [1, 32, 8192, 128] (64, 90) [2784] / 2806        [4, 16, 8192, 128] (64, 90) [5475] / 5580        [1, 3, 4096, 64] (32, 58) [90] / 101
    //   two heads   [1, 2, 8192, 128] (64, 90) 213 / [188]           [1, 2, 6000, 128] (47, 73) 155 / [139]           [1, 2, 4096, 128] (32, 50) [83] / 92
    // Written over keys or values that dQ reads, dK and dV come last.
    const int q_tiles = Tpad / kBlk, window_tiles = (p.window < Tpad ? p.window : Tpad) / kBlk + 2;
    const long long longest = (long long)(p.n[1] > 0 || p.n[2] > 0 || q_tiles < window_tiles ? q_tiles : window_tiles) * p.kv_group;
    const long long causal_tiles = ((long long)p.q_offset + Tpad + kBlk - 1) / kBlk;
    const long long dq_longest = (long long)(p.kv_tiles[0] < window_tiles ? p.kv_tiles[0] : window_tiles) +
                                 (p.kv_tiles[1] < causal_tiles ? p.kv_tiles[1] : causal_tiles) + p.kv_tiles[2];
    const bool longer = 12 * longest > 13 * dq_longest, two_heads = (long long)p.B * p.H <= 2 && q_tiles >= 40;
    p.dq_first = p.dkv_items == 0 || bp.in_place || longest < 24 || p.dkv_items + p.dq_items <= 148 || !(longer || two_heads);
    p.dG = p.dq_first && !bp.dg_last && p.dkv_items > 0 ? bp.dG : nullptr;
    auto launch_dq = [&] {
        e = cudaFuncSetAttribute(bwd_dq_tc_kernel<DH>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::kSmemDq);
        if (e == cudaSuccess) e = launch_chained(bwd_dq_tc_kernel<DH>, dim3((unsigned)(p.dq_items < 148 ? p.dq_items : 148)), dim3(C::kThreads), C::kSmemDq, st, 0, m, p);
    };
    if (p.dq_first) launch_dq();
    if (e == cudaSuccess && p.dkv_items > 0) {
        e = cudaFuncSetAttribute(bwd_dkv_tc_kernel<DH>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::kSmemDkv);
        const long long ctas = p.dkv_items + (!p.dG ? 0 : (long long)p.B * p.T * 3 + C::kThreadsDkv - 1) / C::kThreadsDkv;   // key tiles and sums of dG
        if (e == cudaSuccess) e = launch_chained(bwd_dkv_tc_kernel<DH>, dim3((unsigned)(ctas < 148 ? ctas : 148)), dim3(C::kThreadsDkv), C::kSmemDkv, st, 0, m, p);
    }
    if (e == cudaSuccess && !p.dq_first) launch_dq();
    return e != cudaSuccess || p.dG ? e : launch_bwd_dgate(bp.Gpart, bp.B, bp.H, bp.T, bp.dG, st);
}

}  // namespace

bool bwd_tc_eligible(const BwdParams& p, int dtype) {
    if (dtype != MKA_BF16) return false;
    if (p.d != 64 && p.d != 128) return false;
    if (p.H > 65535 || p.B > 65535) return false;
    for (int l = 0; l < 3; ++l) {
        const LevelDev& L = p.L[l];
        if (L.n == 0) continue;
        if (L.n > 0x7fffffffLL - 256) return false;
        if (L.sn % 8 || L.sn <= 0) return false;
        if (p.H / (p.kv_group > 0 ? p.kv_group : 1) > 1 && (L.sh % 8 || L.sh <= 0)) return false;
        if (p.B > 1 && (L.sb % 8 || L.sb <= 0)) return false;
        if (p.dL[l].sn % 8 || p.dL[l].sh % 8 || p.dL[l].sb % 8) return false;
    }
    return tensor_map_encoder_available();
}

cudaError_t launch_bwd_tc(const BwdParams& p, unsigned int* status_word, cudaStream_t st) {
    if (p.B == 0 || p.H == 0 || p.T == 0) return cudaSuccess;
    return p.d == 128 ? launch_t<128>(p, status_word, st) : launch_t<64>(p, status_word, st);
}

}  // namespace mka

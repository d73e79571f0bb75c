// Tensor-core forward of Eq. 5 for bf16 on sm_100a: TMA -> shared memory -> tcgen05.mma -> TMEM.
//
// A CTA works on a block: 128-row query tiles -- two of them ("ping" and "pong": 256 rows of a head, or 128 rows of two heads of
// a group) at d = 128, one at d = 64, where two CTAs share an SM -- and ONE level-ordered list of 128-row key tiles: all
// visible L1 tiles, then L2, then L3.  A single running (max, sum) per row spans the three levels (the max shift of
// Eq. 11-14); the gate enters as a per-row, per-level additive bias log2(lambda) inside the exponent, so that
//     p = 2^(s * tau * log2(e) + log2(lambda_l) - m)  =  lambda_l * exp(s*tau - m')
// which is exactly the gated, un-normalised weight of Eq. 5.  One normalisation at the end.
//
// Warp roles (d = 128: 384 threads, d = 64: 256):
//   softmax warps    four per query tile, thread = one query row (TMEM lane) x 128 key columns.  Reads S from TMEM, applies
//                    bias and masks, running max, exp2, packs the weights to bf16 and writes them to TMEM in parts of
//                    32 keys (at d = 128 over the columns S occupied), rescales the O accumulator when the running
//                    maximum grows by more than 2^8 (lazy rescale), and does the epilogue.
//   next warp        producer: the warp waits converged, one lane issues the TMA loads of Q and of the K / V tile list
//                    into 128-byte-swizzled shared-memory rings (one mbarrier pair per stage); with paged levels every
//                    lane issues its own box.
//   next warp        issues every tcgen05.mma (the warp runs its loop converged, one elected lane issues):
//                    S_q = Q_q K^T (both operands from shared memory) and O_q += P_q V (P from TMEM, V from shared
//                    memory, N-major) in pieces that follow the parts of P, so that most of the product runs under the
//                    remaining exponentials.  At d = 128 the order is  S0(e)  O1(e-1)  S1(e)  O0(e):  each tile's
//                    softmax overlaps the other tile's products.
//   next warp        deals: works out the CTA's items (blocks, or pieces of their tile lists).
//   last warp        idle: it completes the last warpgroup, so that registers can be moved from it to the softmax
//                    warpgroups (setmaxnreg): a launch leaves 168 (d = 64, two CTAs per SM: 128) registers per thread.
// TMEM: S tiles first (128 columns each), then the O accumulators (d columns each); at d = 64 a P region of 64 columns
// per query tile follows, and S_q(e+1) is multiplied while the softmax of S_q(e) runs (the hand-off is "S is in
// registers", not "P has been consumed").  d = 128 uses all 512 columns, d = 64 256.
// What bounds the d = 128 kernel is the chain  softmax_q(e) -> O_q += P V -> S_q(e+1) -> softmax_q(e+1):  a key tile
// costs the tensor pipe 2048 cycles and the special-function unit 2048 cycles for the two query tiles, but S_q(e+1)
// cannot be written before P_q(e), which lies over S_q(e), has been consumed, and TMEM has no room for a second S.
// A key tile of 256 query rows takes 1.5 us at 1.8 GHz.  Whatever lengthens the softmax lengthens the chain: with the
// scores held in 168 registers a thread spilled, and the level loop indexed its ranges in local memory: 1.63 us, and
// [1, 32, 8192, 128] (window 2048, 2048 slots) took 1024 us against 946.
// Every mbarrier wait is bounded by a wall-clock limit; on expiry the CTA raises a flag in shared
// memory, writes the device status word, lets every role drain, frees TMEM and returns.
#include <atomic>

#include "tc_ptx.cuh"

namespace mka {
namespace {

constexpr uint32_t kPanelBytes = 128 * 128;          // [128 rows][64 bf16] with 128-byte rows
constexpr float kRescaleThreshold = 8.0f;            // log2 units

struct TcMaps {
    CUtensorMap q;
    CUtensorMap k[3];
    CUtensorMap v[3];
};

struct TcParams {
    __nv_bfloat16* O;
    float* LSE;
    const float* gate;
    long long n[3];
    int B, H, T;
    int kv_group;            // query heads per KV head
    int window, q_offset;
    float scale_log2;
    unsigned int* status;
    unsigned long long wait_limit_ns;
    int test_stall;          // test hook (MKA_FLAG_TEST_STALL): the producer leaves out the last key tile of every CTA
    // paged levels: a 128-row key tile is assembled from boxes of box_rows rows, one page-table look-up per box
    int paged;
    const int* table[3];
    long long table_stride[3], table_head_stride[3];
    int page_shift[3], box_rows[3], pool_pages[3];
    const int* rows[3];      // per-sequence rows of a level (clamped to [0, n]), or null
    int deal;                // lines per group of blocks dealt by query block (1 = line by line)
    // A block = query tiles that walk one key-tile list.  d = 64: one tile.  d = 128: two, either 256 consecutive rows of one head, or
    // (pair_heads) the same 128 rows of two heads that share a KV head.  A "line" = what the blocks of one column of rows belong
    // to: a (batch, head), or a (batch, pair of heads).
    int pair_heads;
    int block_rows;          // rows that a block moves down by: 128 or 256
    int lines, q_blocks;     // lines, and blocks of one
    int line_units;          // kStream: units of one line
    int range, longer;       // kStream: units of a CTA's range; the first `longer` CTAs have one more
    float* slots;            // kStream: two partial results per CTA
};

template <int DH>
struct Cfg {
    // A softmax thread owns a whole query row (128 key columns).  d = 128: one CTA per SM with two query tiles (all 512 TMEM
    // columns).  d = 64: the scores of one key tile cost the special-function unit as much as at d = 128 but only half the
    // tensor work, and the tile lists of the training shapes are short; there a CTA takes ONE query tile (256 TMEM
    // columns) and two CTAs share the SM, so that one CTA's waits and epilogue run under the other's steady state.  With
    // two threads to a row (64 columns each, sixteen softmax warps on the SM) the exchange of the row maximum put a barrier of
    // all eight warps into every tile: [8, 16, 2048, 64] (window 512, 1024 slots) took 288 us against 258.
    static constexpr int kNumQ = DH == 128 ? 2 : 1;
    static constexpr int kCtasPerSm = DH == 128 ? 1 : 2;
    static constexpr int kMergeCols = DH == 128 ? 16 : 8;      // columns of a row that a thread merges at a time (kCluster)
    static constexpr int kParts = kTileN / 32;                // the weights of a tile are handed over in parts of 32 keys
    // d = 64 sums the weights of keys 0..63 and 64..127 of a tile apart, each with a running sum of its own: in one chain of
    // all 128 small weights are lost beside large ones earlier (64 weights of 2^-24 after four of 1: LSE short by 9.5e-7 of 1.39, now by a rounding; [8, 16, 2048,
    // 64] on normal inputs: LSE off by 4.45e-8 in one chain, 4.42e-8 in two).  The parts are taken from the two halves in turn, which adds up O's products
    // in the order of the sums.
    static constexpr int kSums = DH == 64 ? 2 : 1;
    static constexpr __host__ __device__ int part_of(int i) { return kSums == 2 && (i == 1 || i == 2) ? 3 - i : i; }
    // A pair of weights in every poly_every()-th group of four is formed on the FMA pipe (exp2_pair_poly, as exact as the special-function unit's):
    // d = 64 keeps that unit busy 84 % of a CTA's steady state, and d = 128 runs at the power cap, where a sixth of the weights on
    // the other pipe cost less than they save.  us, none / every 8th / 4th / 3rd / 2nd group / every group:
    //   [1, 32, 32768, 128] whole blocks    12,747 / 12,747 / 12,550 / [12,400] / 12,383 / 13,785      [8, 16, 2048, 64]    272 / 268 / [269] / 269 / 268 / 320
    //   [4, 16, 8192, 128]                  1777 / 1744 / 1740 / [1724] / 1720 / 1913                  [1, 16, 777, 64]     22.2 / 22.1 / [21.8] / 21.8 / 21.7 / -
    // (whole blocks of 30 to 2000 us at d = 128: 0.96 to 1.00 of the time without; over paged levels, which give the dense form's bits, every 3rd 0.98 to
    // 1.00, every 2nd up to 1.02).  Cut lists at d = 128 (clusters, equal ranges) end before the power cap is reached, and there the longer chain
    // shows: a 512-row chunk at 15,000 rows of context 150.7, with every 3rd group 152.6, every 2nd 157.6.
    static constexpr __host__ __device__ int poly_every(int form) { return DH == 64 ? 4 : (form == 0 ? 3 : 0); }
    static constexpr int kRowWarps = 4;                       // softmax warps per query tile
    static constexpr int kSoftmaxWarps = kRowWarps * kNumQ;
    // The registers are re-divided between the warpgroups (setmaxnreg, a warpgroup-wide instruction: an idle warp
    // completes the last one).  A thread's 128 scores need more than the 168 (d = 64: 128) registers that a launch gives.
    static constexpr int kThreads = (kSoftmaxWarps + 4) * 32;
    static constexpr int kProducerWarp = kSoftmaxWarps, kMmaWarp = kSoftmaxWarps + 1, kDealWarp = kSoftmaxWarps + 2;
    // What the warpgroups hold after the move must not exceed what the launch gave the CTA, or the increase would
    // wait forever:  d = 128: 384 threads x 168 registers at launch = 256 x 216 + 128 x 72;  d = 64: 256 x 128 = 128 x 200 + 128 x 56.
    static constexpr int kRegsLaunch = DH == 128 ? 168 : 128, kRegsSoftmax = DH == 128 ? 216 : 200, kRegsOther = DH == 128 ? 72 : 56;
    static_assert(kSoftmaxWarps * 32 * kRegsSoftmax + 4 * 32 * kRegsOther <= kThreads * kRegsLaunch, "register pool of the CTA exceeded");
    static_assert(kThreads * kCtasPerSm * (kRegsLaunch + 8) > 65536, "the launch would get more than kRegsLaunch registers per thread");
    static constexpr int kPanels = DH / 64;
    static constexpr uint32_t kTileBytes = kPanels * kPanelBytes;
    static constexpr int kStages = 2;
    static constexpr uint32_t kSmemBytes = (kNumQ + 2 * kStages) * kTileBytes + 1024;
    static constexpr uint32_t kIdescQK = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kTileN >> 3) << 17) | ((uint32_t)(kTileM >> 4) << 24);
    // With d = 64 the O accumulator leaves TMEM columns free: P gets a region of its own there instead of
    // overwriting S, so S(e+1) can be multiplied while the softmax of S(e) is still running.
    static constexpr bool kSeparateP = DH == 64;
    static constexpr uint32_t kColO = kNumQ * kTileN;          // first accumulator column (S tiles come first)
    static constexpr uint32_t kColP = kColO + kNumQ * DH;     // first P column when kSeparateP
    static constexpr uint32_t kTmemCols = DH == 128 ? 512u : 256u;
    static_assert(kColP + (kSeparateP ? kNumQ * (kTileN / 2) : 0) <= kTmemCols, "TMEM columns exceeded");
    static constexpr uint32_t kIdescPV = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((uint32_t)(DH >> 3) << 17) | ((uint32_t)(kTileM >> 4) << 24);
    static constexpr int kSlotFloats = kNumQ * kTileM * (DH + 2);   // a partial result of a block: O as [columns / 4][rows][4], then (max, sum) of every row
};

constexpr int kMaxQ = 2;
constexpr int kMaxSplit = 8;              // CTAs of a cluster (the portable limit)


struct Barriers {
    uint64_t q_full;
    uint64_t k_full[4], k_empty[4], v_full[4], v_empty[4];
    uint64_t s_full[kMaxQ], p_part[kMaxQ][4], pv_done[kMaxQ];   // p_part: that part of 32 keys is written
    uint64_t s_free[kMaxQ];   // d = 64 only: the warpgroup has read S(e) into registers, S(e+1) may overwrite it
    uint64_t q_empty;         // the item's Q tiles have had their last reader
    uint64_t item_full[2], item_free[2];
};

// A block of query rows, or a part of its key-tile list, with the rows of the levels it sees.
struct Item {
    int b, kvh, E;            // E: key tiles; -1: there is no further item
    int slot;                 // where the partial result goes; -1: the item is a whole block
    int h[kMaxQ], m[kMaxQ];   // head and first row of each query tile
    int first[3], end[3], n[3];
};

// Key-tile range [first, end) of a block of query rows [r0, r1] (inclusive) on one level.
__host__ __device__ __forceinline__ void tile_range(int level, long long r0, long long r1, int q_offset, int window, long long n,
                                           int& first, int& end) {
    long long lo_f, hi_f, lo_l, hi_l;
    visible_range(level, r0 + q_offset, window, n, 0, lo_f, hi_f);
    visible_range(level, r1 + q_offset, window, n, 0, lo_l, hi_l);
    const long long hi = hi_l > hi_f ? hi_l : hi_f;
    if (hi <= lo_f) { first = end = 0; return; }
    first = (int)(lo_f / kTileN);
    end = (int)((hi + kTileN - 1) / kTileN);
}

// N (a multiple of 8) consecutive columns of one row as bf16.
template <int N>
__device__ __forceinline__ void store_cols_bf16(__nv_bfloat16* out, const float (&x)[N]) {
#pragma unroll
    for (int c = 0; c < N; c += 8) {
        uint4 v;
        v.x = pack_bf16(x[c], x[c + 1]); v.y = pack_bf16(x[c + 2], x[c + 3]);
        v.z = pack_bf16(x[c + 4], x[c + 5]); v.w = pack_bf16(x[c + 6], x[c + 7]);
        *reinterpret_cast<uint4*>(out + c) = v;
    }
}

// How the work is dealt to the CTAs:
//   kWhole    a CTA takes one block of query rows.
//   kCluster  the CTAs of a cluster share one block and split its key-tile list between them (see form_rule).  Each ends with its
//             own un-normalised O and (max, sum); they meet in distributed shared memory, so no scratch memory is needed.
//   kStream   the key tiles of all blocks, laid end to end, are cut into equal ranges, one per resident CTA.  A CTA works off the pieces of
//             blocks in its range one after the other: the next piece's copies and first products run under the epilogue of
//             the one before.  Pieces of cut blocks go to scratch memory and fwd_merge_kernel adds them up.
enum { kWhole = 0, kCluster = 1, kStream = 2 };
constexpr int kStreamRounds = 4;    // kStream is looked at up to this many rounds of resident CTAs
constexpr int kBlockUnits = 2;      // kStream: a block counts as its key tiles and this many more (its epilogue)

// Units of block `qb` of every line.
__host__ __device__ __forceinline__ int block_units(int qb, int rows, int T, int q_offset, int window, const long long (&n)[3]) {
    const long long r0 = (long long)qb * rows, r1 = r0 + rows - 1;
    int units = kBlockUnits;
#pragma unroll
    for (int l = 0; l < 3; ++l) {
        int first = 0, end = 0;
        if (n[l] > 0) tile_range(l, r0, r1 < T - 1 ? r1 : T - 1, q_offset, window, n[l], first, end);
        units += end - first;
    }
    return units;
}

// Heads and first rows of the query tiles of block qb of a line.  A tile without a partner head starts past the last row.
template <int DH>
__device__ __forceinline__ void block_tiles_of(const TcParams& p, int line, int qb, int& b, int& kvh, int (&h)[kMaxQ], int (&m)[kMaxQ]) {
    const int H_kv = p.H / p.kv_group;
    if (DH == 128 && p.pair_heads) {
        const int per = (p.kv_group + 1) / 2, bk = line / per, j = 2 * (line - bk * per);
        b = bk / H_kv; kvh = bk - b * H_kv;
        h[0] = kvh * p.kv_group + j;
        m[0] = qb * kTileM;
        h[1] = j + 1 < p.kv_group ? h[0] + 1 : h[0];
        m[1] = j + 1 < p.kv_group ? m[0] : p.T;
        return;
    }
    b = line / p.H;
    h[0] = h[1] = line - b * p.H;
    kvh = h[0] / p.kv_group;
    m[0] = qb * Cfg<DH>::kNumQ * kTileM;
    m[1] = m[0] + kTileM;
}

// kStream: first unit of CTA i's range, and the CTA whose range holds unit u.
__device__ __forceinline__ int range_start(const TcParams& p, int i) { return i * p.range + min(i, p.longer); }
__device__ __forceinline__ int range_of(const TcParams& p, int u) {
    const int head = p.longer * (p.range + 1);
    return u < head ? u / (p.range + 1) : p.longer + (u - head) / p.range;
}

// Block that holds unit u of a line, and its first unit.  Called by a whole warp.
__device__ __forceinline__ void find_block(const TcParams& p, int u, int lane, int& qb, int& unit0) {
    int before = 0;
    for (int q0 = 0;; q0 += 32) {
        const int own = q0 + lane < p.q_blocks ? block_units(q0 + lane, p.block_rows, p.T, p.q_offset, p.window, p.n) : 0;
        int sum = own;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int x = __shfl_up_sync(0xffffffffu, sum, o);
            if (lane >= o) sum += x;
        }
        const unsigned int past = __ballot_sync(0xffffffffu, before + sum > u);
        if (past || q0 + 32 >= p.q_blocks) {
            const int i = past ? __ffs(past) - 1 : min(31, p.q_blocks - 1 - q0);
            qb = q0 + i;
            unit0 = before + __shfl_sync(0xffffffffu, sum - own, i);
            return;
        }
        before += __shfl_sync(0xffffffffu, sum, 31);
    }
}

template <int DH, bool kPaged, int kForm>
__global__ void __launch_bounds__(Cfg<DH>::kThreads, Cfg<DH>::kCtasPerSm) fwd_tc_kernel(const __grid_constant__ TcMaps maps, const TcParams p) {
    using C = Cfg<DH>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    uint8_t* sQ = smem;                                   // C::kNumQ tiles
    uint8_t* sK = sQ + C::kNumQ * C::kTileBytes;             // kStages tiles
    uint8_t* sV = sK + C::kStages * C::kTileBytes;        // kStages tiles
    __shared__ Barriers bar;
    __shared__ uint32_t tmem_base_slot;
    __shared__ WaitCtl wait_ctl;
    __shared__ Item items[2];
    __shared__ float cl_max[kForm == kCluster ? C::kNumQ : 1][kTileM], cl_sum[kForm == kCluster ? C::kNumQ : 1][kTileM];   // this CTA's (max, sum) of every row, for its cluster

    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // tid >> 5, but provably warp-uniform for the compiler
    int crank = 0, csize = 1;                                 // this CTA's place in its cluster
    if constexpr (kForm == kCluster) {
        asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(crank));
        asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(csize));
    }
    // The whole block `qb` of a line.
    auto block_of = [&](int line, int qb, Item& it) {
        block_tiles_of<DH>(p, line, qb, it.b, it.kvh, it.h, it.m);
        it.slot = -1; it.E = 0;
        const long long m_last = min((long long)it.m[0] + p.block_rows - 1, (long long)p.T - 1);
#pragma unroll
        for (int l = 0; l < 3; ++l) {
            long long n = p.n[l];
            if (kPaged && p.rows[l]) {                        // rows of the level for this sequence
                const long long r = p.rows[l][it.b];
                n = r < 0 ? 0 : (r < n ? r : n);
            }
            it.n[l] = (int)n;
            if (n > 0) tile_range(l, it.m[0], m_last, p.q_offset, p.window, n, it.first[l], it.end[l]);
            else it.first[l] = it.end[l] = 0;
            it.E += it.end[l] - it.first[l];
        }
    };
    // Tiles [t0, t1) of the level-ordered list.
    auto cut = [&](Item& it, int t0, int t1) {
        int base = 0;
        it.E = 0;
#pragma unroll
        for (int l = 0; l < 3; ++l) {
            const int cnt = it.end[l] - it.first[l];
            const int a = min(max(t0 - base, 0), cnt), z = min(max(t1 - base, 0), cnt);
            it.end[l] = it.first[l] + z;
            it.first[l] += a;
            it.E += z - a;
            base += cnt;
        }
    };
    // kStream: the next piece of this CTA's range [u, u1) that holds tiles (or the start of a block without tiles).
    int u = 0, u1 = 0, unit0 = 0;                             // unit0: first unit of block (line, qb)  (fewer than 2^30 units)
    int line = 0, qb = 0;
    auto next_piece = [&](Item& it) {
        while (u < u1) {
            block_of(line, qb, it);
            const int E = it.E;
            const int t0 = u - unit0, t1 = min(E, u1 - unit0);
            u = unit0 + E + kBlockUnits;
            unit0 = u;
            if (++qb == p.q_blocks) { qb = 0; ++line; }
            if (E == 0 ? t0 > 0 : t0 >= t1) continue;         // nothing but the block's epilogue, which goes with its last tile
            if (t0 > 0 || t1 < E) {
                cut(it, t0, t1);
                it.slot = 2 * (int)blockIdx.x + (t0 > 0 ? 0 : 1);
            }
            return;
        }
        it.E = -1;
    };

    if (tid == 0) {
        wait_ctl.abort = 0;
        wait_ctl.limit_ns = p.wait_limit_ns;
        mbar_init(&bar.q_full, 1);
        for (int s = 0; s < 4; ++s) {
            mbar_init(&bar.k_full[s], 1); mbar_init(&bar.k_empty[s], 1);
            mbar_init(&bar.v_full[s], 1); mbar_init(&bar.v_empty[s], 1);
        }
        for (int q = 0; q < C::kNumQ; ++q) {
            mbar_init(&bar.s_full[q], 1); mbar_init(&bar.pv_done[q], 1);
            for (int i = 0; i < 4; ++i) mbar_init(&bar.p_part[q][i], C::kRowWarps);   // one arrival per softmax warp
            mbar_init(&bar.s_free[q], C::kRowWarps);
        }
        mbar_init(&bar.q_empty, 1);
        for (int i = 0; i < 2; ++i) { mbar_init(&bar.item_full[i], 1); mbar_init(&bar.item_free[i], 2 + C::kSoftmaxWarps); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    auto first_item = [&] {
        Item it;
        if constexpr (kForm == kStream) {
            u = range_start(p, blockIdx.x); u1 = range_start(p, blockIdx.x + 1);
            line = u / p.line_units;
            int in_line;
            find_block(p, u - line * p.line_units, lane, qb, in_line);
            unit0 = line * p.line_units + in_line;
            next_piece(it);
        } else {
            // Blocks start in the order of their linear index.  Within a group of p.deal lines the blocks are
            // dealt by query block, heaviest (latest rows) first for every line of the group, then the next lighter one: the
            // launch then ends with the group's lightest blocks instead of the last head's heaviest.
            const int lin = (int)blockIdx.x / csize;          // fewer than 2^31 blocks
            const int per_group = p.deal * p.q_blocks;
            const int grp = lin / per_group, in_grp = lin - grp * per_group;
            const int lines_here = min(p.deal, p.lines - grp * p.deal);
            block_of(grp * p.deal + in_grp % lines_here, p.q_blocks - 1 - in_grp / lines_here, it);
            if constexpr (kForm == kCluster) {                // this CTA's share of the list
                const int total = it.E;
                cut(it, (int)((long long)total * crank / csize), (int)((long long)total * (crank + 1) / csize));
            }
        }
        if (lane == 0) items[0] = it;
    };
    chain_trigger();
    if (kForm == kStream && warp == C::kDealWarp) first_item();              // (from the call's arguments alone)
    chain_wait();
    if (kForm != kStream && warp == C::kDealWarp) first_item();
    // The status word starts at OK.  CTAs start in the order of their numbers and none gives up before the wait limit (100 us at
    // least) has passed, so the first one clears it before any other can have something to report.
    if (tid == 0 && (blockIdx.x | blockIdx.y | blockIdx.z) == 0) atomicExch(p.status, (unsigned int)MKA_OK);
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_slot)), "r"(C::kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base_slot;
    volatile WaitCtl* abortp = &wait_ctl;

    // Item number i is in items[i & 1]: the first from the start, the others once the dealing warp has posted them.  A warp that
    // is done with one says so.
    auto has_item = [&](int i) -> bool {
        if (i > 0) {
            if (kForm != kStream || !mbar_wait_warp(&bar.item_full[i & 1], (uint32_t)((i - 1) >> 1) & 1u, abortp)) return false;
        }
        return items[i & 1].E >= 0;
    };
    auto done_item = [&](int i) {
        if constexpr (kForm == kStream) {
            __syncwarp();
            if (lane == 0) mbar_arrive(&bar.item_free[i & 1]);
        }
    };

    if (warp >= C::kSoftmaxWarps) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(C::kRegsOther));
    if (warp == C::kProducerWarp) {
        // The warp waits converged.  Dense levels: one lane issues (inside an `if (lane == 0)` around the whole loop the
        // kernel keeps its loop state in local memory: 1.63 us per key tile instead of 1.49 at d = 128).
        // Paged levels: the whole warp produces.  Lane i owns box i of every key tile (a box = the rows of one page
        // that fall into the tile): it looks its page up while the warp waits for the stage to drain and issues its
        // own copies, so a tile costs one table round trip (overlapped) and four warp-wide copy instructions.
        int issued = 0, it = 0;                               // key tiles and items
        bool ok = true;
        for (; ok && has_item(it); ++it) {
            const Item& I = items[it & 1];
            const int b = I.b, kvh = I.kvh;
            if (it > 0 && !mbar_wait_warp(&bar.q_empty, (uint32_t)(it - 1) & 1u, abortp)) break;
            if (lane == 0) {
                mbar_expect_tx(&bar.q_full, C::kNumQ * C::kTileBytes);
#pragma unroll
                for (int q = 0; q < C::kNumQ; ++q)
#pragma unroll
                    for (int pn = 0; pn < C::kPanels; ++pn)
                        tma_load_4d(sQ + q * C::kTileBytes + pn * kPanelBytes, &maps.q, pn * 64, I.m[q], I.h[q], b, &bar.q_full);
            }
            __syncwarp();
            int left = I.E;
#pragma unroll 1
            for (int l = 0; l < 3 && ok; ++l) {
                const int kt_first = I.first[l], kt_end = I.end[l];
                if (kt_first >= kt_end) continue;
                const long long n_here = I.n[l];
                const int* tab = kPaged ? p.table[l] + (long long)b * p.table_stride[l] + (long long)kvh * p.table_head_stride[l] : nullptr;
                const int rpb = kPaged ? p.box_rows[l] : kTileN;
                const bool mine = lane < kTileN / rpb;
                const int in_mask = kPaged ? (1 << p.page_shift[l]) - 1 : 0;
                for (int kt = kt_first; kt < kt_end; ++kt) {
                    // test hook: the item's last tile never arrives (kStream: of the first item in one half of the CTAs, of the second in the other)
                    if (!kPaged && p.test_stall && it == (kForm == kStream ? (int)(blockIdx.x & 1) : 0) && --left == 0) { ok = false; break; }
                    const int s = issued % C::kStages;
                    const uint32_t ph = (uint32_t)(issued / C::kStages) & 1u;
                    // a box past the level's last row is aimed past the pool, where the copy engine fills zeros as it does
                    // past a dense level's end
                    int z = kt * kTileN, w = b;                        // dense: row in the level, batch; paged: row in the page, page
                    if constexpr (kPaged) {
                        const long long row = (long long)kt * kTileN + lane * rpb;
                        w = p.pool_pages[l];
                        if (mine && row < n_here) w = tab[row >> p.page_shift[l]];
                        z = (int)(row & in_mask);
                    }
                    if (!mbar_wait_warp(&bar.k_empty[s], ph ^ 1u, abortp)) { ok = false; break; }
                    if (lane == 0) mbar_expect_tx(&bar.k_full[s], C::kTileBytes);
                    __syncwarp();
                    if (mine) {
#pragma unroll
                        for (int pn = 0; pn < C::kPanels; ++pn)
                            tma_load_4d(sK + s * C::kTileBytes + pn * kPanelBytes + lane * rpb * 128, &maps.k[l], pn * 64, z, kvh, w, &bar.k_full[s]);
                    }
                    __syncwarp();
                    if (!mbar_wait_warp(&bar.v_empty[s], ph ^ 1u, abortp)) {           // gave up with this stage's K copies in flight
                        mbar_drain(&bar.k_full[s], ph, abortp, gtimer());
                        ok = false;
                        break;
                    }
                    if (lane == 0) mbar_expect_tx(&bar.v_full[s], C::kTileBytes);
                    __syncwarp();
                    if (mine) {
#pragma unroll
                        for (int pn = 0; pn < C::kPanels; ++pn)
                            tma_load_4d(sV + s * C::kTileBytes + pn * kPanelBytes + lane * rpb * 128, &maps.v[l], pn * 64, z, kvh, w, &bar.v_full[s]);
                    }
                    __syncwarp();
                    ++issued;
                }
            }
            if (!ok) { ++it; break; }                         // its Q was asked for
            done_item(it);
        }
        // Before leaving, make sure every copy issued has landed (bounded): the shared memory must not be handed to
        // another CTA with a bulk copy still in flight.  (A stage whose wait failed got no copies.)
        const unsigned long long t_drain = gtimer();
        if (it > 0) mbar_drain(&bar.q_full, (uint32_t)(it - 1) & 1u, abortp, t_drain);
        for (int i = issued > C::kStages ? issued - C::kStages : 0; i < issued; ++i) {
            mbar_drain(&bar.k_full[i % C::kStages], (uint32_t)(i / C::kStages) & 1u, abortp, t_drain);
            mbar_drain(&bar.v_full[i % C::kStages], (uint32_t)(i / C::kStages) & 1u, abortp, t_drain);
        }
    } else if (warp == C::kDealWarp) {
        if constexpr (kForm == kStream) {
            for (int it = 1;; ++it) {
                Item next;
                next_piece(next);
                // This wait lasts as long as the work on item it - 2, which is in the way: some waits of the other roles for each of its key
                // tiles, and it is allowed as many limits.  Should one of those run out, it ends this one.  (Counting the tiles as they
                // are asked for and starting the clock again with each cost a 512-row chunk at 15,000 rows of context 1.5 %.)
                if (it >= 2 && !mbar_wait_warp(&bar.item_free[it & 1], (uint32_t)((it - 2) >> 1) & 1u, abortp, 8u * (items[it & 1].E + 1))) break;
                if (lane == 0) {
                    items[it & 1] = next;
                    mbar_arrive(&bar.item_full[it & 1]);
                }
                __syncwarp();
                if (next.E < 0) break;
            }
        }
    } else if (warp == C::kMmaWarp) {
        {   // every lane runs the issue loop (converged); elect.sync inside the wrappers picks the issuing lane
            // low descriptor words of the operands (see make_desc)
            const uint32_t q_lo = desc_lo_kmajor(smem_u32(sQ)), k_lo = desc_lo_kmajor(smem_u32(sK));
            const uint32_t v_lo = desc_lo_mnmajor(smem_u32(sV), kPanelBytes);
            auto issue_qk = [&](int q, int s) {
                const uint32_t qa = q_lo + q * (C::kTileBytes >> 4), ka = k_lo + s * (C::kTileBytes >> 4);
#pragma unroll
                for (int k = 0; k < DH / 16; ++k)
                    mma_ss_elect(tmem + q * kTileN, make_desc(qa + kstep_off(k, kPanelBytes)), make_desc(ka + kstep_off(k, kPanelBytes)),
                           C::kIdescQK, k > 0);
                mma_commit_elect(&bar.s_full[q]);
            };
            auto k_ready = [&](int g) { return mbar_wait_warp(&bar.k_full[g % C::kStages], (uint32_t)(g / C::kStages) & 1u, abortp); };
            auto v_ready = [&](int g) { return mbar_wait_warp(&bar.v_full[g % C::kStages], (uint32_t)(g / C::kStages) & 1u, abortp); };
            // O_q += P_q V in parts: the softmax warps hand over the weights of 32 keys at a time (K-steps 2 part,
            // 2 part + 1), so that the product runs under the remaining exponentials.
            auto issue_pv = [&](int q, int g, bool accumulate) -> bool {
                const uint32_t va = v_lo + (g % C::kStages) * (C::kTileBytes >> 4);
                const uint32_t pa = tmem + (C::kSeparateP ? C::kColP + q * (kTileN / 2) : q * kTileN);
#pragma unroll
                for (int n = 0; n < C::kParts; ++n) {
                    if (!mbar_wait_warp(&bar.p_part[q][C::part_of(n)], (uint32_t)g & 1u, abortp)) return false;
                    tc_fence_after();
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        const int k = C::part_of(n) * 2 + i;
                        mma_ts_elect(tmem + C::kColO + q * DH, pa + k * 8, make_desc(va + k * (2048 >> 4)), C::kIdescPV,
                                     (accumulate || n > 0 || i > 0) ? 1u : 0u);
                    }
                }
                mma_commit_elect(&bar.pv_done[q]);
                return true;
            };
            int g = 0;                                        // key tiles of the CTA, across its items
            bool ok = true;
            for (int it = 0; ok && has_item(it); ++it) {
            const Item& I = items[it & 1];
            const int E = __shfl_sync(0xffffffffu, I.E, 0);   // warp-uniform for the compiler too
            // Paged levels: the page that holds a level's last row is copied whole, so the rows after that row arrive
            // with whatever the pool holds there (a recycled page, never-written memory).  Their weights are exactly 0,
            // but 0 x NaN or 0 x Inf would still poison the accumulator: those V rows are cleared here, after the
            // copy has landed and before the product reads them.  (K needs nothing: masked scores are overwritten.)
            int scrub_e[3] = {-1, -1, -1}, scrub_r0[3] = {0, 0, 0}, scrub_r1[3] = {0, 0, 0};
            if (kPaged) {
                int e0 = 0;
#pragma unroll
                for (int l = 0; l < 3; ++l) {
                    const int tiles = I.end[l] - I.first[l];
                    const int tail = I.n[l] % kTileN;
                    if (tiles > 0 && tail != 0 && (long long)I.end[l] * kTileN > I.n[l]) {
                        const int rpb = p.box_rows[l];
                        scrub_e[l] = e0 + tiles - 1;
                        scrub_r0[l] = tail;
                        scrub_r1[l] = (tail + rpb - 1) / rpb * rpb;      // end of the box that straddles the level's end
                    }
                    e0 += tiles;
                }
            }
            auto scrub_v = [&](int e, int s) {
                if constexpr (kPaged) {
#pragma unroll
                for (int l = 0; l < 3; ++l) {
                    if (e != scrub_e[l]) continue;
                    const int vecs = (scrub_r1[l] - scrub_r0[l]) * 8;      // 16-byte vectors per 64-column panel
                    for (int pn = 0; pn < C::kPanels; ++pn) {
                        uint4* base = reinterpret_cast<uint4*>(sV + s * C::kTileBytes + pn * kPanelBytes + scrub_r0[l] * 128);
                        for (int i = lane; i < vecs; i += 32) base[i] = make_uint4(0u, 0u, 0u, 0u);
                    }
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                }
                }
            };
            if (!(ok = mbar_wait_warp(&bar.q_full, (uint32_t)it & 1u, abortp))) break;
            tc_fence_after();
            if (E == 0) {
                mma_commit_elect(&bar.q_empty);
                done_item(it);
                continue;
            }
            if (!(ok = k_ready(g))) break;
            if (C::kSeparateP) {
                // S_q(e+1) is issued as soon as the warpgroup has S_q(e) in registers; O_q += P_q(e) V(e) when P_q(e) is written.
                for (int q = 0; q < C::kNumQ && ok; ++q) {
                    if (g > 0 && !mbar_wait_warp(&bar.s_free[q], (uint32_t)(g - 1) & 1u, abortp)) { ok = false; break; }
                    tc_fence_after();
                    issue_qk(q, g % C::kStages);
                }
                if (!ok) break;
                mma_commit_elect(&bar.k_empty[g % C::kStages]);
                if (E == 1) mma_commit_elect(&bar.q_empty);
                for (int e = 0; e < E && ok; ++e, ++g) {
                    const int s = g % C::kStages, sn = (g + 1) % C::kStages;
                    if (e + 1 < E) {
                        if (!k_ready(g + 1)) { ok = false; break; }
#pragma unroll
                        for (int q = 0; q < C::kNumQ; ++q) {
                            if (!mbar_wait_warp(&bar.s_free[q], (uint32_t)g & 1u, abortp)) { ok = false; break; }
                            tc_fence_after();
                            issue_qk(q, sn);
                        }
                        if (!ok) break;
                        mma_commit_elect(&bar.k_empty[sn]);
                        if (e + 2 == E) mma_commit_elect(&bar.q_empty);
                    }
                    if (!v_ready(g)) { ok = false; break; }
                    scrub_v(e, s);
#pragma unroll
                    for (int q = 0; q < C::kNumQ; ++q) {
                        if (!issue_pv(q, g, e > 0)) { ok = false; break; }
                    }
                    if (!ok) break;
                    mma_commit_elect(&bar.v_empty[s]);
                }
            } else {
                // The wait for K(e+1) is taken before the wait for P_0(e), so that S_0(e+1) follows O_0(e) at once: that
                // pair of products is what query tile 0's softmax threads are waiting for.
                for (int e = 0; e < E && ok; ++e, ++g) {
                    const int s = g % C::kStages;
                    tc_fence_after();
                    issue_qk(0, s);
                    if (e > 0) {
                        if (!issue_pv(1, g - 1, e - 1 > 0)) { ok = false; break; }
                        mma_commit_elect(&bar.v_empty[(g - 1) % C::kStages]);
                    }
                    issue_qk(1, s);
                    mma_commit_elect(&bar.k_empty[s]);
                    if (e + 1 == E) mma_commit_elect(&bar.q_empty);
                    if (!v_ready(g)) { ok = false; break; }
                    scrub_v(e, s);
                    if (e + 1 < E && !k_ready(g + 1)) { ok = false; break; }
                    if (!issue_pv(0, g, e > 0)) { ok = false; break; }
                }
                if (!ok) break;
                if (!(ok = issue_pv(1, g - 1, E > 1))) break;
                mma_commit_elect(&bar.v_empty[(g - 1) % C::kStages]);
            }
            done_item(it);
            }
        }
    }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(C::kRegsSoftmax));
        // ------------------------------------------------------------ softmax warps
        // warp = (query tile, lane quarter); thread = one query row (TMEM lane)
        const int q = warp / C::kRowWarps;
        const int row_in_tile = (warp & 3) * 32 + lane;
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t s_addr = tmem + lane_base + q * kTileN;
        const uint32_t o_addr = tmem + lane_base + C::kColO + q * DH;
        // where this thread's weights go as bf16 pairs
        const uint32_t p_addr = C::kSeparateP ? tmem + lane_base + C::kColP + q * (kTileN / 2) : tmem + lane_base + q * kTileN;
        bool ok = true;                                                          // warp-uniform
        int g = 0;                                                               // key tiles of the CTA, across its items
#pragma unroll 1
        for (int it = 0; ok && has_item(it); ++it) {
        const Item& I = items[it & 1];
        const int tq0 = I.m[q];                                                  // first row of this query tile
        const int t = tq0 + row_in_tile;                                         // T < 2^31 - 256
        const bool row_valid = t < p.T;
        float m_run = -INFINITY, l_part[C::kSums] = {};
        int e = 0;
#pragma unroll 1
        for (int l = 0; l < 3 && ok; ++l) {
            const int kt_first = I.first[l], kt_end = I.end[l];
            if (kt_first == kt_end) continue;
            const long long n_here = I.n[l];
            float bias = -INFINITY;
            int lo = 0, hi = 0;                              // visible rows of this level (levels hold fewer than 2^31 rows)
            // A row past T has a bias of -inf, so its weights are 0 whatever it sees: it takes the last row's range and
            // costs its warp no mask of its own.
            if (row_valid) {
                const float gt = p.gate[((long long)I.b * p.T + t) * 3 + l];
                bias = gt > 0.f ? log2f(gt) : -INFINITY;
            }
            // key tiles visible to every row of THIS query tile need no element mask
            int full_first = 0, full_end = 0x7fffffff;                     // (a tile without a row inside T masks nothing)
            if (tq0 < p.T) {
                const int tq1 = min(tq0 + kTileM - 1, p.T - 1);
                {
                    long long lo64, hi64;
                    visible_range(l, (row_valid ? (long long)t : tq1) + p.q_offset, p.window, n_here, 0, lo64, hi64);
                    lo = (int)lo64; hi = (int)hi64;
                }
                long long lo_f, hi_f, lo_l, hi_l;
                visible_range(l, (long long)tq0 + p.q_offset, p.window, n_here, 0, lo_f, hi_f);
                visible_range(l, (long long)tq1 + p.q_offset, p.window, n_here, 0, lo_l, hi_l);
                full_first = (int)((lo_l + kTileN - 1) / kTileN);
                full_end = (int)(hi_f / kTileN);
            }
            for (int kt = kt_first; kt < kt_end; ++kt, ++e, ++g) {
                if (!(ok = __all_sync(0xffffffffu, mbar_wait(&bar.s_full[q], (uint32_t)g & 1u, abortp)))) break;
                float s[kTileN];
                tc_fence_after();
#pragma unroll
                for (int c0 = 0; c0 < kTileN; c0 += 32) tmem_ld32(s_addr + c0, reinterpret_cast<uint32_t*>(s) + c0);
                tmem_ld_wait();
                if (C::kSeparateP) {                         // S(e) is in registers: its TMEM columns may be reused
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&bar.s_free[q]);
                }
                const bool need_mask = !(kt >= full_first && kt < full_end);
                if (need_mask) {
                    const long long col0 = (long long)kt * kTileN;
                    const int c_lo = (int)max(0LL, min((long long)lo - col0, (long long)kTileN));
                    const int c_hi = (int)max(0LL, min((long long)hi - col0, (long long)kTileN));
                    // One bit per column: the bits of 32 columns come from two shifts and each costs a test and a select.
                    // Two comparisons per column made a masked tile take 3.6 us against 1.6 (now 2.1).
#pragma unroll
                    for (int c0 = 0; c0 < kTileN; c0 += 32) {        // 32 columns that no row of the warp masks are passed over
                        const uint32_t vis = low_bits(c_hi - c0) & ~low_bits(c_lo - c0);
                        if (__all_sync(0xffffffffu, vis == 0xffffffffu)) continue;
#pragma unroll
                        for (int i = 0; i < 32; ++i) s[c0 + i] = (vis >> i) & 1u ? s[c0 + i] : -INFINITY;
                    }
                }
                float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
                for (int c = 0; c < kTileN; c += 8) {
                    mx4[0] = max3_nan(mx4[0], s[c], s[c + 1]); mx4[1] = max3_nan(mx4[1], s[c + 2], s[c + 3]);
                    mx4[2] = max3_nan(mx4[2], s[c + 4], s[c + 5]); mx4[3] = max3_nan(mx4[3], s[c + 6], s[c + 7]);
                }
                const float mx = max3_nan(max3_nan(mx4[0], mx4[1], mx4[2]), mx4[3], mx4[3]);
                const float x_row = fmaf(mx, p.scale_log2, bias);            // -inf when the whole row is masked
                // A score of NaN is taken for +inf: from here on the row's weights are 0 or NaN in every column, whatever forms them, its sum is
                // not above 0, and the row ends as O = 0 with LSE = -inf, as one with a score of +inf does.
                const float x_max = x_row == x_row ? x_row : INFINITY;
                const float m_new = fmaxf(m_run, x_max);
                const bool grow = m_new > m_run + kRescaleThreshold;         // also true for the first finite max
                const float m_use = grow ? m_new : m_run;
                const float m_eff = m_use == -INFINITY ? 0.f : m_use;
                const float alpha = grow ? (m_run == -INFINITY ? 0.f : ex2(m_run - m_use)) : 1.f;
                const float shift = bias - m_eff;
#pragma unroll
                for (int i = 0; i < C::kSums; ++i) l_part[i] *= alpha;
                m_run = m_use;
                // P(e-1) must have been consumed before P(e) replaces it (d = 64), and before O is rescaled
                const bool rescale = e > 0 && __any_sync(0xffffffffu, alpha != 1.f);
                if ((C::kSeparateP || rescale) && e > 0) {
                    if (!(ok = __all_sync(0xffffffffu, mbar_wait(&bar.pv_done[q], (uint32_t)(g - 1) & 1u, abortp)))) break;
                    tc_fence_after();
                }
                if (rescale) {                               // some row of this warp moved its reference maximum
#pragma unroll 1
                    for (int c0 = 0; c0 < DH; c0 += 32) {
                        uint32_t o[32];
                        tmem_ld32(o_addr + c0, o);
                        tmem_ld_wait();
#pragma unroll
                        for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * alpha);
                        tmem_st32(o_addr + c0, o);
                    }
                }
                // The weights leave in parts of 32 columns (16 packed pairs, one store each).  A part is handed to
                // the issuing warp in the middle of the next part's exponentials, when its store has long completed.
                // Scale, shift and the row sum work on packed pairs: one instruction for two columns.
                const uint64_t scale2 = pack2(p.scale_log2, p.scale_log2), shift2 = pack2(shift, shift);
                uint64_t sum_a[C::kSums], sum_b[C::kSums];
#pragma unroll
                for (int i = 0; i < C::kSums; ++i) sum_a[i] = sum_b[i] = pack2(0.f, 0.f);
                uint32_t pk[16];
                constexpr int kPoly = C::poly_every(kForm);
                auto weights = [&](int c_from, int c_to, int c_base) {
                    const int half = C::kSums == 2 ? c_base / 64 : 0;
#pragma unroll
                    for (int c = c_from; c < c_to; c += 4) {
                        float x0, x1, x2, x3;
                        unpack2(fma2(pack2(s[c], s[c + 1]), scale2, shift2), x0, x1);
                        unpack2(fma2(pack2(s[c + 2], s[c + 3]), scale2, shift2), x2, x3);
                        const float p0 = ex2(x0), p1 = ex2(x1);
                        float p2, p3;
                        if (kPoly && (c / 4) % (kPoly ? kPoly : 1) == 0) exp2_pair_poly(x2, x3, p2, p3);
                        else p2 = ex2(x2), p3 = ex2(x3);
                        sum_a[half] = add2(sum_a[half], pack2(p0, p1));
                        sum_b[half] = add2(sum_b[half], pack2(p2, p3));
                        pk[(c - c_base) / 2] = pack_bf16(p0, p1);
                        pk[(c - c_base) / 2 + 1] = pack_bf16(p2, p3);
                    }
                };
                auto hand_over = [&](int part) {             // the part (and a rescaled accumulator) is in TMEM
                    tmem_st_wait();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&bar.p_part[q][part]);
                };
#pragma unroll
                for (int n = 0; n < C::kParts; ++n) {
                    const int part = C::part_of(n);
                    weights(32 * part, 32 * part + 16, 32 * part);
                    if (n > 0) hand_over(C::part_of(n - 1));
                    weights(32 * part + 16, 32 * part + 32, 32 * part);
                    tmem_st16(p_addr + 16 * part, pk);
                }
#pragma unroll
                for (int i = 0; i < C::kSums; ++i) {
                    float a0, a1;
                    unpack2(add2(sum_a[i], sum_b[i]), a0, a1);
                    l_part[i] += a0 + a1;
                }
                hand_over(C::part_of(C::kParts - 1));
            }
        }
        const float l_run = C::kSums == 2 ? l_part[0] + l_part[C::kSums - 1] : l_part[0];
        // ------------------------------------------------------------ epilogue
        const int E = I.E;
        if (ok && E > 0) ok = __all_sync(0xffffffffu, mbar_wait(&bar.pv_done[q], (uint32_t)(g - 1) & 1u, abortp));
        if constexpr (kForm == kCluster) {
            // Every operand tile has been read when all softmax warps have seen their last product (and no copy is in
            // flight then), so O may lie over the K and V rings: four columns of all 128 rows, then the next four.
            const bool any = ok && E > 0;
            cl_max[q][row_in_tile] = any ? m_run : -INFINITY;
            cl_sum[q][row_in_tile] = any ? l_run : 0.f;
            asm volatile("bar.sync 4, %0;" ::"n"(C::kSoftmaxWarps * 32) : "memory");
            if (ok && !abortp->abort) {
                tc_fence_after();
                float4* so = reinterpret_cast<float4*>(sK) + q * DH / 4 * kTileM + row_in_tile;
#pragma unroll 1
                for (int c0 = 0; c0 < DH; c0 += 32) {
                    uint32_t o[32];
                    if (E > 0) {
                        tmem_ld32(o_addr + c0, o);
                        tmem_ld_wait();
                    } else {
#pragma unroll
                        for (int i = 0; i < 32; ++i) o[i] = 0u;
                    }
#pragma unroll
                    for (int i = 0; i < 32; i += 4)
                        so[(c0 + i) / 4 * kTileM] = make_float4(__uint_as_float(o[i]), __uint_as_float(o[i + 1]), __uint_as_float(o[i + 2]), __uint_as_float(o[i + 3]));
                }
            }
        } else if (kForm == kStream && ok && I.slot >= 0) {
            // a piece of a cut block: its accumulator as it is, rows next to each other (a warp stores 512 bytes at a time)
            tc_fence_after();
            float* slot = p.slots + (long long)I.slot * C::kSlotFloats;
            float4* so = reinterpret_cast<float4*>(slot) + q * DH / 4 * kTileM + row_in_tile;
#pragma unroll 1
            for (int c0 = 0; c0 < DH; c0 += 32) {
                uint32_t o[32];
                tmem_ld32(o_addr + c0, o);
                tmem_ld_wait();
#pragma unroll
                for (int i = 0; i < 32; i += 4)
                    so[(c0 + i) / 4 * kTileM] = make_float4(__uint_as_float(o[i]), __uint_as_float(o[i + 1]), __uint_as_float(o[i + 2]), __uint_as_float(o[i + 3]));
            }
            reinterpret_cast<float2*>(slot + C::kNumQ * kTileM * DH)[q * kTileM + row_in_tile] = make_float2(m_run, l_run);
        } else if (ok) {
            tc_fence_after();
            const float inv = l_run > 0.f ? 1.f / l_run : 0.f;           // rows with nothing visible: exact zeros
            const int first_row = (warp & 3) * 32;                       // of this warp, within the query tile
            const long long bh = (long long)I.b * p.H + I.h[q];
            __nv_bfloat16* out = p.O + (bh * p.T + tq0 + first_row) * DH;
            const int rows_here = max(0, min(32, p.T - tq0 - first_row));
#pragma unroll 1
            for (int c0 = 0; c0 < DH; c0 += 32) {
                uint32_t o[32];
                if (E > 0) {
                    tmem_ld32(o_addr + c0, o);
                    tmem_ld_wait();
                }
                if (E == 0 || !(inv > 0.f)) {
#pragma unroll
                    for (int i = 0; i < 32; ++i) o[i] = 0u;
                }
                store_rows_bf16<32>(out + c0, DH, rows_here, o, inv, lane);
            }
            if (row_valid && p.LSE) p.LSE[bh * p.T + t] = l_run > 0.f ? (m_run + log2f(l_run)) * kLn2 : -INFINITY;
        }
        done_item(it);
        }
    }

    if constexpr (kForm == kCluster) {
        // Merge: every CTA takes its share of the block's columns, a few at a time, and adds the cluster's parts with the
        // weights 2^(max_i - max) / sum.  The second barrier keeps a CTA's shared memory alive until all have read it.
        __syncwarp();
        cluster_sync();
        if (warp < C::kSoftmaxWarps) {
            const int row_in_tile = (warp & 3) * 32 + lane;
            const uint32_t so = smem_u32(sK) + row_in_tile * 16;
            float w[kMaxSplit];
            int have_q = -1;
            for (int u = crank * (C::kSoftmaxWarps / 4) + (warp >> 2); u < C::kNumQ * DH / C::kMergeCols; u += csize * (C::kSoftmaxWarps / 4)) {
                const int q = u / (DH / C::kMergeCols), c0 = (u % (DH / C::kMergeCols)) * C::kMergeCols;
                const int t = items[0].m[q] + row_in_tile;
                const long long bh = (long long)items[0].b * p.H + items[0].h[q];
                if (t >= p.T) continue;
                if (q != have_q || c0 == 0) {
                    float mi[kMaxSplit], mx = -INFINITY, sum = 0.f;
#pragma unroll
                    for (int i = 0; i < kMaxSplit; ++i) {
                        mi[i] = i < csize ? ld_cluster(smem_u32(&cl_max[q][row_in_tile]), i) : -INFINITY;
                        mx = fmaxf(mx, mi[i]);
                    }
#pragma unroll
                    for (int i = 0; i < kMaxSplit; ++i) {
                        w[i] = mi[i] == -INFINITY ? 0.f : ex2(mi[i] - mx);
                        if (i < csize) sum = fmaf(w[i], ld_cluster(smem_u32(&cl_sum[q][row_in_tile]), i), sum);
                    }
                    const float inv = sum > 0.f ? 1.f / sum : 0.f;       // rows with nothing visible: exact zeros
#pragma unroll
                    for (int i = 0; i < kMaxSplit; ++i) w[i] = inv > 0.f ? w[i] * inv : 0.f;
                    have_q = inv > 0.f ? q : kMaxQ + q;
                    if (c0 == 0 && p.LSE) p.LSE[bh * p.T + t] = sum > 0.f ? (mx + log2f(sum)) * kLn2 : -INFINITY;
                }
                float acc[C::kMergeCols];
#pragma unroll
                for (int c = 0; c < C::kMergeCols; ++c) acc[c] = 0.f;
                if (have_q == q) {
#pragma unroll
                    for (int i0 = 0; i0 < kMaxSplit; i0 += 2) {          // the loads of two parts are in flight together
                        if (i0 >= csize) break;
                        const int i1 = i0 + 1 < csize ? i0 + 1 : i0;      // (an odd last part is read twice and added once)
                        float4 o[2][C::kMergeCols / 4];
#pragma unroll
                        for (int c = 0; c < C::kMergeCols; c += 4) {
                            o[0][c / 4] = ld_cluster4(so + (q * DH + c0 + c) / 4 * (kTileM * 16), i0);
                            o[1][c / 4] = ld_cluster4(so + (q * DH + c0 + c) / 4 * (kTileM * 16), i1);
                        }
#pragma unroll
                        for (int i = 0; i < 2; ++i) {
                            if (i0 + i >= csize) continue;
#pragma unroll
                            for (int c = 0; c < C::kMergeCols; c += 4) {
                                acc[c] = fmaf(w[i0 + i], o[i][c / 4].x, acc[c]); acc[c + 1] = fmaf(w[i0 + i], o[i][c / 4].y, acc[c + 1]);
                                acc[c + 2] = fmaf(w[i0 + i], o[i][c / 4].z, acc[c + 2]); acc[c + 3] = fmaf(w[i0 + i], o[i][c / 4].w, acc[c + 3]);
                            }
                        }
                    }
                }
                store_cols_bf16<C::kMergeCols>(p.O + (bh * p.T + t) * DH + c0, acc);
            }
        }
        __syncwarp();
        cluster_sync();
    }
    tc_fence_before();
    __syncthreads();
    if (tid == 0 && wait_ctl.abort) atomicExch(p.status, (unsigned int)MKA_ERR_TIMEOUT);
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(C::kTmemCols) : "memory");
}

// kStream, second kernel: adds up the pieces of the cut blocks.  Boundary i = blockIdx.x + 1 lies between the ranges of CTAs i - 1 and i
// of the first kernel; the first boundary inside a block's tiles does the whole block, eight columns of 128 rows to a warpgroup.
// Its bytes come from the L2 cache: two pieces of 128 KB (d = 128) at most per CTA.
constexpr int kMergeThreads = 256, kMergeAhead = 4;
template <int DH>
__global__ void __launch_bounds__(kMergeThreads, 4) fwd_merge_kernel(const TcParams p) {
    using C = Cfg<DH>;
    chain_trigger();
    const int lane = threadIdx.x & 31;
    const int cut = range_start(p, blockIdx.x + 1);                       // first unit of CTA blockIdx.x + 1
    const int line = cut / p.line_units;
    int qb, unit0;
    find_block(p, cut - line * p.line_units, lane, qb, unit0);
    const int E = block_units(qb, p.block_rows, p.T, p.q_offset, p.window, p.n) - kBlockUnits;
    const int at = line * p.line_units + unit0;                           // the block's first unit
    chain_wait();                                                         // (every CTA: what follows this kernel relies on it for the first one too)
    if (cut <= at || cut >= at + E) return;                               // between two blocks
    const int i0 = range_of(p, at), parts = range_of(p, at + E - 1) - i0 + 1;
    if (i0 != (int)blockIdx.x) return;                                    // not the block's first boundary
    int b, kvh, h[kMaxQ], m[kMaxQ];
    block_tiles_of<DH>(p, line, qb, b, kvh, h, m);
    // CTA i0 holds the block's first tiles in its second slot, the others theirs in their first
    const float* s0 = p.slots + (long long)(2 * i0 + 1) * C::kSlotFloats;
    const long long step = 2LL * C::kSlotFloats;
    const int row = threadIdx.x & 127;
    for (int c8 = blockIdx.y * (kMergeThreads / 128) + (threadIdx.x >> 7); c8 < C::kNumQ * DH / 8; c8 += gridDim.y * (kMergeThreads / 128)) {
    const int q = c8 / (DH / 8), c0 = (c8 % (DH / 8)) * 8;
    const int t = (q == 0 ? m[0] : m[1]) + row;
    if (t >= p.T) continue;
    const int ml_at = C::kNumQ * kTileM * DH + (q * kTileM + row) * 2, o_at = ((q * DH + c0) / 4 * kTileM + row) * 4;
    float mx = -INFINITY, sum = 0.f, acc[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) acc[c] = 0.f;
    for (int i = 0; i < parts; i += kMergeAhead) {                        // the loads of several pieces are in flight together
        float2 ml[kMergeAhead];
        float4 lo[kMergeAhead], hi[kMergeAhead];
#pragma unroll
        for (int j = 0; j < kMergeAhead; ++j) {
            const int k = min(i + j, parts - 1);
            const float* sl = k == 0 ? s0 : s0 + k * step - C::kSlotFloats;
            ml[j] = *reinterpret_cast<const float2*>(sl + ml_at);
            lo[j] = *reinterpret_cast<const float4*>(sl + o_at);
            hi[j] = *reinterpret_cast<const float4*>(sl + o_at + kTileM * 4);
        }
#pragma unroll
        for (int j = 0; j < kMergeAhead; ++j) {
            if (i + j >= parts || ml[j].x == -INFINITY) continue;         // (a row that sees none of the piece's tiles)
            const float m_new = fmaxf(mx, ml[j].x);
            const float keep = mx == -INFINITY ? 0.f : ex2(mx - m_new), w = ex2(ml[j].x - m_new);
            mx = m_new;
            sum = fmaf(w, ml[j].y, sum * keep);
            const float v[8] = {lo[j].x, lo[j].y, lo[j].z, lo[j].w, hi[j].x, hi[j].y, hi[j].z, hi[j].w};
#pragma unroll
            for (int c = 0; c < 8; ++c) acc[c] = fmaf(w, v[c], acc[c] * keep);
        }
    }
    const float inv = sum > 0.f ? 1.f / sum : 0.f;
#pragma unroll
    for (int c = 0; c < 8; ++c) acc[c] = inv > 0.f ? acc[c] * inv : 0.f;
    const long long at_row = ((long long)b * p.H + (q == 0 ? h[0] : h[1])) * p.T + t;
    store_cols_bf16<8>(p.O + at_row * DH + c0, acc);
    if (c0 == 0 && p.LSE) p.LSE[at_row] = sum > 0.f ? (mx + log2f(sum)) * kLn2 : -INFINITY;
    }
}

inline bool make_map(CUtensorMap* map, const void* base, int d, long long rows, int H, int B, long long sn, long long sh, long long sb) {
    return make_bf16_map(map, base, d, rows, H, B, sn, sh, sb, 128);
}

template <int DH>
cudaLaunchConfig_t cluster_config(int split, dim3 grid, cudaStream_t st, cudaLaunchAttribute* at) {
    at->id = cudaLaunchAttributeClusterDimension;
    at->val.clusterDim.x = split; at->val.clusterDim.y = 1; at->val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = grid; cfg.blockDim = dim3(Cfg<DH>::kThreads); cfg.dynamicSmemBytes = Cfg<DH>::kSmemBytes; cfg.stream = st;
    cfg.attrs = at; cfg.numAttrs = 1;
    return cfg;
}

// A kernel of the forward's shape (threads, shared memory) and CTAs per SM, asked about in its place: for a kernel that moves registers
// between its warps the occupancy query finds one CTA to an SM at d = 64, where two run (112 clusters of two CTAs, which it
// takes for two rounds of 74, end after 15.8 us; a whole block of theirs after 18.3).
template <int DH>
__global__ void __launch_bounds__(Cfg<DH>::kThreads, Cfg<DH>::kCtasPerSm) fwd_shape_kernel() {}

// Clusters of `split` CTAs that the device keeps resident at a time (a cluster stays within one GPC, so this is less than
// the number of CTAs / split); asked once per device and size.
template <int DH>
int resident_clusters(int split) {
    static std::atomic<int> known[64][kMaxSplit + 1];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    int n = known[dev][split].load(std::memory_order_relaxed);
    if (n) return n - 1;
    auto kern = fwd_shape_kernel<DH>;
    cudaLaunchAttribute at;
    const cudaLaunchConfig_t cfg = cluster_config<DH>(split, dim3(split), nullptr, &at);
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg<DH>::kSmemBytes) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;                                             // not split this time; only answers are remembered
    }
    known[dev][split].store(n + 1, std::memory_order_relaxed);
    return n;
}

// How the query tiles are put into blocks.
struct Blocks {
    int pair_heads, rows;         // see TcParams
    long long lines;
    int per_line;
};

// Key tiles of one block (device row counts of paged levels are not known here: n bounds them).
int block_tiles(const FwdParams& fp, const Blocks& bl, long long q_block) {
    const long long n[3] = {fp.L[0].n, fp.L[1].n, fp.L[2].n};
    return block_units((int)q_block, bl.rows, fp.T, fp.q_offset, fp.window, n) - kBlockUnits;
}

// d = 128: 256 consecutive rows of a head, or 128 rows of two heads of a group where that makes fewer key tiles to walk (a last
// block with 128 rows or fewer is half empty; two heads see exactly the same keys).  2 x 69 rows at 5467, 32 heads on 8, in
// clusters, the better size for each: 82 us in blocks of one head, 49 in pairs.
template <int DH>
Blocks make_blocks(const FwdParams& fp) {
    Blocks bl;
    bl.pair_heads = 0; bl.rows = Cfg<DH>::kNumQ * kTileM;
    bl.lines = (long long)fp.B * fp.H;
    bl.per_line = (fp.T + bl.rows - 1) / bl.rows;
    if (DH != 128 || fp.kv_group < 2 || bl.per_line > 32) return bl;
    Blocks two = {1, kTileM, bl.lines / fp.kv_group * ((fp.kv_group + 1) / 2), (fp.T + kTileM - 1) / kTileM};
    double t1 = 0.0, t2 = 0.0;
    for (int i = 0; i < bl.per_line; ++i) t1 += block_tiles(fp, bl, i) + kBlockUnits;
    for (int i = 0; i < two.per_line; ++i) t2 += block_tiles(fp, two, i) + kBlockUnits;
    return t2 * (double)two.lines < 0.97 * t1 * (double)bl.lines ? two : bl;
}

// Which form.  A launch whose blocks do not fill the chip, or fill it a little more than once, leaves SMs idle while others walk whole
// lists.  Cluster or equal ranges then share the lists out; the first costs its merge and whole clusters per GPC, the second a pass
// of partial results through the L2 cache, and its CTAs, each in another place of the keys, find less of them there.  All are added
// up in us: a round of resident CTAs lasts as long as its first (heaviest) block.  The constants were fitted to 34 sizes (8 to 1600
// blocks, 4 to 490 tiles a block), over which the pick takes 0.7 % more than the best form on average, and for d = 64 again to 40, where it took
// 3.2 % more with one cluster CTA counted to an SM, now 1.5 % (CTAs of clusters share SMs from about 96 on).  Whole / clusters of 2 / 3 /
// 4 / 8 / ranges, chosen in brackets:
//   d = 128, 28 heads on 4, 512 rows at 15,000 rows of context      265 / 144 / 195 / 155 / 191 / [124] us   (56 blocks, 160 tiles)
//   d = 128, 12 on 4, 949 rows at 3804                              93 / 59 / 79 / 69 / 101 / [51] us        (48 blocks, 61 tiles)
//   d = 128, 12 on 4, 175 rows at 4662                              90 / 53 / 40 / 34 / [25] / 33 us         (12 blocks, 54 tiles)
//   d = 128, 12 on 4, 124 rows at 36,735                            452 / 234 / 161 / 124 / 73 / [55] us     (8 blocks, 295 tiles)
//   d = 128, 32 on 8, 2 x 69 rows at 5467                           127 / 83 / 58 / [49] / 84 / 63 us        (32 blocks, 75 tiles)
//   d = 128, 16 heads, 3078 rows                                    164 / 170 / 194 / 228 / 347 / [155] us   (208 blocks)
//   d = 128, 2 x 16 heads, 1000 rows                                [35] / 51 / 63 / 80 / 149 / 56 us        (128 blocks)
//   d = 64, 2 x 32 heads, 627 rows, 7815 slots                      179 / 157 / 159 / 164 / 205 / [137] us   (320 blocks)
//   d = 64, 16 heads, 777 rows                                      19 / [17] / 23 / 24 / 41 / 21 us         (112 blocks)
//   d = 64, 32 heads on 8, 479 rows, 1698 slots                     29 / [25] / 34 / 32 / 51 / 30 us         (128 blocks)
struct FormChoice { int form, ctas; };       // kCluster: CTAs of a cluster; kStream: CTAs of the grid
template <int DH>
FormChoice form_rule(const FwdParams& fp, const Blocks& bl, bool scratch) {
    const long long lines = bl.lines, blocks = lines * bl.per_line;
    const int slots = 148 * Cfg<DH>::kCtasPerSm;
    const double tile = DH == 128 ? 1.54 : 0.93;                            // us for a CTA that has its SM to itself
    const double whole_first = DH == 128 ? 7.0 : 6.5, whole_next = DH == 128 ? 4.5 : 3.0;           // a round's start and end
    const double cluster_first = DH == 128 ? 14.5 : 9.2, cluster_next = DH == 128 ? 11.5 : 9.0;
    const double cluster_tile = DH == 128 ? 1.03 : 1.1;
    const double ranges_first = DH == 128 ? 17.5 : 16.5, ranges_tile = DH == 128 ? 1.18 : 1.14;
    auto shared = [](long long ctas, long long sms = 148) { return DH == 64 && ctas > sms ? 1.28 : 1.0; };
    FormChoice best = {kWhole, 1};
    if (blocks > kStreamRounds * slots) return best;                         // whole blocks fill the chip evenly enough
    double best_us = 0.0;
    for (long long blk = 0; blk < blocks; blk += slots)
        best_us += block_tiles(fp, bl, bl.per_line - 1 - blk / lines) * tile * shared(blocks - blk) + (blk == 0 ? whole_first : whole_next);
    best_us *= 0.97;                                                         // (what the model can tell apart)
    if (blocks <= slots) {
        for (int split = 2; split <= kMaxSplit; ++split) {
            // d = 64: three tiles to a CTA at least (2 x 16 heads on 4, 220 rows, 5 tiles: 11.2 us whole, 13.9 in clusters of 4)
            if (DH == 64 && 3 * split > block_tiles(fp, bl, bl.per_line - 1)) break;
            const int fit = resident_clusters<DH>(split);
            if (fit < 1) continue;
            double us = 0.0;
            for (long long blk = 0; blk < blocks && us < best_us; blk += fit)
                us += block_tiles(fp, bl, bl.per_line - 1 - blk / lines) * tile * cluster_tile / split * shared((blocks - blk < fit ? blocks - blk : fit) * split, 96) +
                      (blk == 0 ? cluster_first : cluster_next);
            if (us < best_us) { best = {kCluster, split}; best_us = us; }
        }
    }
    if (scratch) {
        double units = 0.0, mbytes = 0.0;
        for (int qb = 0; qb < bl.per_line; ++qb) units += block_tiles(fp, bl, qb) + kBlockUnits;
        units *= (double)lines;
        for (int l = 0; l < 3; ++l) {
            const double seen = l == 0 ? (double)fp.window + fp.T : 1e18;
            mbytes += ((double)fp.L[l].n < seen ? (double)fp.L[l].n : seen) * fp.B * (fp.H / fp.kv_group) * (DH * 4e-6);
        }
        const double us = units / slots * tile * ranges_tile * shared(slots) + ranges_first + 0.35 * slots / (double)blocks + (mbytes > 100.0 ? 0.068 * (mbytes - 100.0) : 0.0);
        if (units >= slots && units < 1e9 && us < best_us) best = {kStream, slots};
    }
    return best;
}

template <int DH>
bool known_rows(const FwdParams& fp) {       // kStream cuts by the levels' lengths, which a row count per sequence may undercut
    for (int l = 0; l < 3; ++l) if (fp.paged && fp.L[l].n > 0 && fp.paged[l].rows) return false;
    return true;
}
template <int DH>
size_t scratch_bytes_t(const FwdParams& fp) {
    const Blocks bl = make_blocks<DH>(fp);
    if (bl.lines * bl.per_line > kStreamRounds * 148 * Cfg<DH>::kCtasPerSm || !known_rows<DH>(fp)) return 0;
    const FormChoice c = form_rule<DH>(fp, bl, true);
    return c.form == kStream ? (size_t)2 * c.ctas * Cfg<DH>::kSlotFloats * sizeof(float) : 0;
}

template <int DH>
cudaError_t launch_t(const FwdParams& fp, unsigned int* status_word, cudaStream_t st) {
    TcMaps maps;
    if (!make_map(&maps.q, fp.Q, DH, fp.T, fp.H, fp.B, DH, (long long)fp.T * DH, (long long)fp.H * fp.T * DH))
        return cudaErrorNotSupported;
    TcParams p;
    memset(&p, 0, sizeof(p));
    p.paged = fp.paged ? 1 : 0;
    for (int l = 0; l < 3; ++l) {
        if (fp.L[l].n == 0) { maps.k[l] = maps.q; maps.v[l] = maps.q; continue; }
        if (fp.paged) {
            // the pool as a [pages, KV heads, rows of a page, d] tensor; a box = (up to 128) rows of one page
            const PagedLevelDev& P = fp.paged[l];
            const int page_rows = 1 << P.page_shift;
            const int rpb = page_rows < kTileN ? page_rows : kTileN;
            if (!make_bf16_map(&maps.k[l], P.k, DH, page_rows, fp.H / fp.kv_group, (int)P.pool_pages, P.sn, P.sh, P.sp, rpb) ||
                !make_bf16_map(&maps.v[l], P.v, DH, page_rows, fp.H / fp.kv_group, (int)P.pool_pages, P.sn, P.sh, P.sp, rpb))
                return cudaErrorNotSupported;
            p.table[l] = P.table; p.table_stride[l] = P.table_stride; p.table_head_stride[l] = P.table_head_stride;
            p.page_shift[l] = P.page_shift; p.box_rows[l] = rpb; p.pool_pages[l] = (int)P.pool_pages; p.rows[l] = P.rows;
            continue;
        }
        if (!make_map(&maps.k[l], fp.L[l].k, DH, fp.L[l].n, fp.H / fp.kv_group, fp.B, fp.L[l].sn, fp.L[l].sh, fp.L[l].sb) ||
            !make_map(&maps.v[l], fp.L[l].v, DH, fp.L[l].n, fp.H / fp.kv_group, fp.B, fp.L[l].sn, fp.L[l].sh, fp.L[l].sb))
            return cudaErrorNotSupported;
    }
    p.O = static_cast<__nv_bfloat16*>(fp.O);
    p.LSE = fp.LSE;
    p.gate = fp.gate;
    for (int l = 0; l < 3; ++l) p.n[l] = fp.L[l].n;
    p.B = fp.B; p.H = fp.H; p.T = fp.T; p.kv_group = fp.kv_group;
    p.window = fp.window; p.q_offset = fp.q_offset;
    p.scale_log2 = fp.scale * kLog2e;
    p.status = status_word;
    p.wait_limit_ns = wait_limit_ns();
    p.test_stall = fp.test_stall;
    const Blocks bl = make_blocks<DH>(fp);
    {   // as many lines per group as keep the group's K and V (48 MB at most) in the L2 cache while
        // its blocks, dealt by query block, re-read them
        double pair_bytes = 0.0;
        for (int l = 0; l < 3; ++l) pair_bytes += (double)fp.L[l].n * DH * 4.0;
        pair_bytes /= bl.pair_heads ? (fp.kv_group + 1) / 2 : fp.kv_group;
        const double lines = (double)bl.lines;
        const double fit = pair_bytes > 0.0 ? 48.0 * 1024 * 1024 / pair_bytes : lines;
        p.deal = fit < 1.0 ? 1 : (fit > lines ? (int)lines : (int)fit);
    }
    p.pair_heads = bl.pair_heads; p.block_rows = bl.rows; p.lines = (int)bl.lines; p.q_blocks = bl.per_line;
    const bool scratch = fp.scratch && (reinterpret_cast<uintptr_t>(fp.scratch) & 15) == 0 && known_rows<DH>(fp);
    FormChoice form = form_rule<DH>(fp, bl, scratch);
    if (form.form == kStream && fp.scratch_bytes < (size_t)2 * form.ctas * Cfg<DH>::kSlotFloats * sizeof(float)) form = form_rule<DH>(fp, bl, false);
    auto kern = form.form == kStream    ? (fp.paged ? fwd_tc_kernel<DH, true, kStream> : fwd_tc_kernel<DH, false, kStream>)
                : form.form == kCluster ? (fp.paged ? fwd_tc_kernel<DH, true, kCluster> : fwd_tc_kernel<DH, false, kCluster>)
                                        : (fp.paged ? fwd_tc_kernel<DH, true, kWhole> : fwd_tc_kernel<DH, false, kWhole>);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg<DH>::kSmemBytes);
    if (e != cudaSuccess) return e;
    const long long blocks = bl.lines * bl.per_line;
    if (form.form != kStream) {
        if (blocks * form.ctas > 0x7fffffffLL) return cudaErrorInvalidValue;
        return launch_chained(kern, dim3((unsigned)(blocks * form.ctas)), dim3(Cfg<DH>::kThreads), Cfg<DH>::kSmemBytes, st,
                              form.form == kCluster ? form.ctas : 0, maps, p);
    }
    for (int qb = 0; qb < bl.per_line; ++qb) p.line_units += block_units(qb, bl.rows, p.T, p.q_offset, p.window, p.n);
    const int units = p.lines * p.line_units;
    p.range = units / form.ctas; p.longer = units % form.ctas;
    p.slots = static_cast<float*>(fp.scratch);
    e = launch_chained(kern, dim3(form.ctas), dim3(Cfg<DH>::kThreads), Cfg<DH>::kSmemBytes, st, 0, maps, p);
    if (e != cudaSuccess) return e;
    return launch_chained(fwd_merge_kernel<DH>, dim3(form.ctas - 1, DH == 128 ? 4 : 2), dim3(kMergeThreads), 0, st, 0, p);
}

}  // namespace

size_t fwd_tc_scratch_bytes(const FwdParams& p) {
    if (p.B == 0 || p.H == 0 || p.T == 0) return 0;
    return p.d == 128 ? scratch_bytes_t<128>(p) : scratch_bytes_t<64>(p);
}

bool fwd_tc_eligible(const FwdParams& p, int dtype) {
    if (dtype != MKA_BF16 || p.mode != MKA_MODE_FAST || p.decode) return false;
    if (p.d != 64 && p.d != 128) return false;
    if (p.H > 65535 || p.B > 65535) return false;
    if ((double)((p.T + 127) / 128) * p.H * p.B > 2147483647.0) return false;   // the kernel numbers its blocks in an int
    for (int l = 0; l < 3; ++l) {
        const LevelDev& L = p.L[l];
        if (L.n == 0) continue;
        if (L.n > 0x7fffffffLL) return false;
        if (L.sn % 8 || L.sn <= 0) return false;
        if (p.H / (p.kv_group > 0 ? p.kv_group : 1) > 1 && (L.sh % 8 || L.sh <= 0)) return false;
        if (p.B > 1 && (L.sb % 8 || L.sb <= 0)) return false;
    }
    return tensor_map_encoder_available();
}

cudaError_t launch_fwd_tc(const FwdParams& p, unsigned int* status_word, cudaStream_t st) {
    if (p.B == 0 || p.H == 0 || p.T == 0) return cudaSuccess;
    return p.d == 128 ? launch_t<128>(p, status_word, st) : launch_t<64>(p, status_word, st);
}

}  // namespace mka

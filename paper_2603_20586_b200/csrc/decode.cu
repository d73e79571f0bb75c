// Split-KV single-token decode of Eq. 5 (all cached rows of the three levels visible).
//
// Two forms (cluster_rule).  Short and evenly dealt caches: one kernel, decode_cluster_kernel, whose clusters finish a (batch, head)
// each.  Otherwise the split form, two kernels; the paged and grouped decode (decode_paged.cu) ends with the second of them:
// Kernel 1 (HBM-bound, streams K and V exactly once): grid = (batch*head) x chunks of the split
// table.  A row of d bf16 values is covered by d/8 lanes with one 16-byte load each, so a warp reads
// 32*16 contiguous bytes per instruction; each lane group keeps its own running (max, sum, acc) in the
// base-2 domain (the max shift of Eq. 11-14) and the groups, then the CTA's warps, are merged with
// warp shuffles / shared memory into one UN-GATED partial per chunk: (m_c, z_c, acc_c[d]).
// Kernel 2: per (batch, head), gate-weighted log-sum-exp combine over all chunks of all levels:
//   O = sum_c lam_{l(c)} 2^{m_c-M} acc_c / sum_c lam_{l(c)} 2^{m_c-M} z_c.
#include <mutex>

#include "tc_ptx.cuh"

namespace mka {
namespace {

constexpr int kWarps = 8;
constexpr int kMaxCluster = 8;   // CTAs of a cluster (the portable limit)
constexpr int kUnroll = 8;   // independent 16-byte loads in flight per lane, per stream (K and V)

__device__ __forceinline__ uint4 ld_stream(const void* p) {
    uint4 r;
    asm volatile("ld.global.nc.L1::no_allocate.L2::128B.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "l"(p));
    return r;
}

__device__ __forceinline__ void unpack8(const uint4& u, float (&x)[8]) {
    const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        x[2 * i] = __uint_as_float(w[i] << 16);
        x[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
    }
}

// Merges the lane groups of a warp (lanes that hold the same column slice).
template <int LPR>
__device__ __forceinline__ void merge_groups(float& m, float& z, float (&acc)[8]) {
#pragma unroll
    for (int o = 16; o >= LPR; o >>= 1) {
        const float m_o = __shfl_xor_sync(0xffffffffu, m, o);
        const float z_o = __shfl_xor_sync(0xffffffffu, z, o);
        const float m_n = fmaxf(m, m_o);
        const float a = m_n > -INFINITY ? exp2f(m - m_n) : 0.f;
        const float c = m_n > -INFINITY ? exp2f(m_o - m_n) : 0.f;
        z = z * a + z_o * c;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float acc_o = __shfl_xor_sync(0xffffffffu, acc[i], o);
            acc[i] = acc[i] * a + acc_o * c;
        }
        m = m_n;
    }
}

// Column threadIdx.x of the CTA's warps together.
template <int DH>
__device__ __forceinline__ void merge_warps(const float (&sm_m)[kWarps], const float (&sm_z)[kWarps], const float (&sm_acc)[kWarps][DH], float& M,
                                            float& Z, float& A) {
    M = -INFINITY;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) M = fmaxf(M, sm_m[w]);
    Z = 0.f; A = 0.f;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
        const float f = M > -INFINITY ? exp2f(sm_m[w] - M) : 0.f;
        Z = fmaf(sm_z[w], f, Z);
        A = fmaf(sm_acc[w][threadIdx.x], f, A);
    }
}

template <int DH>
__global__ void __launch_bounds__(kWarps * 32, 2) decode_partial_kernel(const DecodeParams p) {
    chain_enter();
    constexpr int LPR = DH / 8;          // lanes per row
    constexpr int RPI = 32 / LPR;        // rows per warp-wide load instruction
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int sub = lane % LPR;          // which 8-column slice of the row this lane holds
    const int grp = lane / LPR;          // which row of the instruction
    const long long bh = blockIdx.x / p.total_chunks;
    long long chunk = blockIdx.x % p.total_chunks;
    int lvl = 0;
    while (lvl < 2 && chunk >= p.n_chunks[lvl]) { chunk -= p.n_chunks[lvl]; ++lvl; }
    const LevelDev L = p.L[lvl];
    const int b = (int)(bh / p.H), h = (int)(bh % p.H);
    const long long r_begin = chunk * p.chunk_rows;
    const long long r_end = r_begin + p.chunk_rows < L.n ? r_begin + p.chunk_rows : L.n;
    if (p.gate[b * 3 + lvl] == 0.f) {                  // hard routing switched this level off: do not read it
        float* out = p.partial + (long long)blockIdx.x * (DH + 2);
        for (int i = threadIdx.x; i < DH + 2; i += kWarps * 32) out[i] = i == 0 ? -INFINITY : 0.f;
        return;
    }
    const __nv_bfloat16* Kp = static_cast<const __nv_bfloat16*>(L.k) + b * L.sb + (h / p.kv_group) * L.sh + sub * 8;
    const __nv_bfloat16* Vp = static_cast<const __nv_bfloat16*>(L.v) + b * L.sb + (h / p.kv_group) * L.sh + sub * 8;

    float q[8];
    {
        uint4 u = *reinterpret_cast<const uint4*>(static_cast<const __nv_bfloat16*>(p.q) + bh * DH + sub * 8);
        unpack8(u, q);
        const float c = p.scale * kLog2e;     // scores in the base-2 domain
#pragma unroll
        for (int i = 0; i < 8; ++i) q[i] *= c;
    }
    float m = -INFINITY, z = 0.f, acc[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[i] = 0.f;

    // rows of this chunk are dealt to warps in slabs of RPI*kUnroll consecutive rows
    constexpr int SLAB = RPI * kUnroll;
    for (long long r0 = r_begin + (long long)warp * SLAB; r0 < r_end; r0 += (long long)kWarps * SLAB) {
        uint4 kk[kUnroll], vv[kUnroll];
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            long long r = r0 + u * RPI + grp;
            long long rc = r < r_end ? r : r_end - 1;        // clamp: a tail lane re-reads the last row
            kk[u] = ld_stream(Kp + rc * L.sn);
        }
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            long long r = r0 + u * RPI + grp;
            long long rc = r < r_end ? r : r_end - 1;
            vv[u] = ld_stream(Vp + rc * L.sn);
        }
        float s[kUnroll];
        float smax = -INFINITY;
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            float x[8];
            unpack8(kk[u], x);
            float d0 = 0.f;
#pragma unroll
            for (int i = 0; i < 8; ++i) d0 = fmaf(q[i], x[i], d0);
#pragma unroll
            for (int o = LPR / 2; o > 0; o >>= 1) d0 += __shfl_xor_sync(0xffffffffu, d0, o);
            const bool ok = r0 + u * RPI + grp < r_end;
            s[u] = ok ? d0 : -INFINITY;
            smax = fmaxf(smax, s[u]);
        }
        const float m_new = fmaxf(m, smax);
        if (m_new > -INFINITY) {
            const float resc = exp2f(m - m_new);             // m = -inf gives 0
            z *= resc;
#pragma unroll
            for (int i = 0; i < 8; ++i) acc[i] *= resc;
#pragma unroll
            for (int u = 0; u < kUnroll; ++u) {
                const float e = exp2f(s[u] - m_new);         // masked rows: exp2(-inf) = 0
                z += e;
                float x[8];
                unpack8(vv[u], x);
#pragma unroll
                for (int i = 0; i < 8; ++i) acc[i] = fmaf(e, x[i], acc[i]);
            }
            m = m_new;
        }
    }

    merge_groups<LPR>(m, z, acc);
    // merge the warps of the CTA
    __shared__ float sm_m[kWarps], sm_z[kWarps], sm_acc[kWarps][DH];
    if (grp == 0) {
#pragma unroll
        for (int i = 0; i < 8; ++i) sm_acc[warp][sub * 8 + i] = acc[i];
        if (sub == 0) { sm_m[warp] = m; sm_z[warp] = z; }
    }
    __syncthreads();
    if (threadIdx.x < DH) {
        float M, Z, A;
        merge_warps<DH>(sm_m, sm_z, sm_acc, M, Z, A);
        float* out = p.partial + (long long)blockIdx.x * (DH + 2);
        out[2 + threadIdx.x] = A;
        if (threadIdx.x == 0) { out[0] = M; out[1] = Z; }
    }
}

// Short caches: ONE kernel.  The CTAs of a cluster share a (batch, head); the slabs of its three levels are dealt over all of
// their warps, the gate enters as log2(gate) in the exponent, and the CTAs' (max, sum, accumulator) meet in distributed
// shared memory.  A split into chunks has nothing to gain there, and the second kernel costs a launch and its latency: one
// sequence with 32 heads and 512 + 1000 + 64 rows took 12.1 us in two kernels, 9.7 here.
template <int DH>
__global__ void __launch_bounds__(kWarps * 32, 2) decode_cluster_kernel(const DecodeParams p) {
    chain_enter();
    constexpr int LPR = DH / 8, RPI = 32 / LPR, SLAB = RPI * kUnroll;
    __shared__ float sm_m[kWarps], sm_z[kWarps], sm_acc[kWarps][DH];
    __shared__ float cta_m, cta_z, cta_acc[DH];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int sub = lane % LPR, grp = lane / LPR;
    int rank, size;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(size));
    const long long bh = blockIdx.x / size;
    const int b = (int)(bh / p.H), h = (int)(bh % p.H);
    float q[8];
    {
        const uint4 u = *reinterpret_cast<const uint4*>(static_cast<const __nv_bfloat16*>(p.q) + bh * DH + sub * 8);
        unpack8(u, q);
        const float c = p.scale * kLog2e;     // scores in the base-2 domain
#pragma unroll
        for (int i = 0; i < 8; ++i) q[i] *= c;
    }
    float lam[3];
    long long end[3];                         // slabs of the levels, running total
#pragma unroll
    for (int l = 0; l < 3; ++l) {
        lam[l] = p.gate[b * 3 + l];
        end[l] = (l ? end[l - 1] : 0) + (p.L[l].n + SLAB - 1) / SLAB;
    }
    float m = -INFINITY, z = 0.f, acc[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[i] = 0.f;
    for (long long slab = (long long)warp * size + rank; slab < end[2]; slab += (long long)kWarps * size) {
        const int l = slab < end[0] ? 0 : (slab < end[1] ? 1 : 2);
        const float g = l == 0 ? lam[0] : (l == 1 ? lam[1] : lam[2]);
        if (!(g > 0.f)) continue;                          // hard routing switched this level off: do not read it
        const LevelDev& L = l == 0 ? p.L[0] : (l == 1 ? p.L[1] : p.L[2]);
        const long long r0 = (slab - (l == 0 ? 0 : (l == 1 ? end[0] : end[1]))) * SLAB;
        const long long base = b * L.sb + (h / p.kv_group) * L.sh + sub * 8;
        const __nv_bfloat16* Kp = static_cast<const __nv_bfloat16*>(L.k) + base;
        const __nv_bfloat16* Vp = static_cast<const __nv_bfloat16*>(L.v) + base;
        uint4 kk[kUnroll], vv[kUnroll];
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            const long long r = r0 + u * RPI + grp;
            kk[u] = ld_stream(Kp + (r < L.n ? r : L.n - 1) * L.sn);        // a tail lane re-reads the last row
        }
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            const long long r = r0 + u * RPI + grp;
            vv[u] = ld_stream(Vp + (r < L.n ? r : L.n - 1) * L.sn);
        }
        const float bias = log2f(g);
        float s[kUnroll], smax = -INFINITY;
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            float x[8];
            unpack8(kk[u], x);
            float d0 = 0.f;
#pragma unroll
            for (int i = 0; i < 8; ++i) d0 = fmaf(q[i], x[i], d0);
#pragma unroll
            for (int o = LPR / 2; o > 0; o >>= 1) d0 += __shfl_xor_sync(0xffffffffu, d0, o);
            s[u] = r0 + u * RPI + grp < L.n ? d0 + bias : -INFINITY;
            smax = fmaxf(smax, s[u]);
        }
        const float m_new = fmaxf(m, smax);
        if (m_new > -INFINITY) {
            const float resc = exp2f(m - m_new);             // m = -inf gives 0
            z *= resc;
#pragma unroll
            for (int i = 0; i < 8; ++i) acc[i] *= resc;
#pragma unroll
            for (int u = 0; u < kUnroll; ++u) {
                const float e = exp2f(s[u] - m_new);         // masked rows: exp2(-inf) = 0
                z += e;
                float x[8];
                unpack8(vv[u], x);
#pragma unroll
                for (int i = 0; i < 8; ++i) acc[i] = fmaf(e, x[i], acc[i]);
            }
            m = m_new;
        }
    }
    merge_groups<LPR>(m, z, acc);
    if (grp == 0) {
#pragma unroll
        for (int i = 0; i < 8; ++i) sm_acc[warp][sub * 8 + i] = acc[i];
        if (sub == 0) { sm_m[warp] = m; sm_z[warp] = z; }
    }
    __syncthreads();
    if (threadIdx.x < DH) {
        float M, Z, A;
        merge_warps<DH>(sm_m, sm_z, sm_acc, M, Z, A);
        cta_acc[threadIdx.x] = A;
        if (threadIdx.x == 0) { cta_m = M; cta_z = Z; }
    }
    cluster_sync();
    // every CTA finishes its share of the columns; the second barrier keeps its shared memory alive for the others
    const int per = (DH + size - 1) / size, c = rank * per + (int)threadIdx.x;
    if ((int)threadIdx.x < per && c < DH) {
        float M = -INFINITY, Z = 0.f, A = 0.f;
        // All reads at once, a missing CTA's from the first one: a branch for each made them follow one another.
        float mi[kMaxCluster], zi[kMaxCluster], ai[kMaxCluster];
#pragma unroll
        for (int i = 0; i < kMaxCluster; ++i) {
            const int from = i < size ? i : 0;
            mi[i] = ld_cluster(smem_u32(&cta_m), from); zi[i] = ld_cluster(smem_u32(&cta_z), from); ai[i] = ld_cluster(smem_u32(&cta_acc[c]), from);
        }
#pragma unroll
        for (int i = 0; i < kMaxCluster; ++i) M = fmaxf(M, mi[i]);
#pragma unroll
        for (int i = 0; i < kMaxCluster; ++i) {
            const float f = i < size && M > -INFINITY ? exp2f(mi[i] - M) : 0.f;
            if (i < size) { Z = fmaf(zi[i], f, Z); A = fmaf(ai[i], f, A); }
        }
        static_cast<__nv_bfloat16*>(p.O)[bh * DH + c] = __float2bfloat16_rn(Z > 0.f ? A / Z : 0.f);
        if (c == 0) {
            if (p.LSE) p.LSE[bh] = Z > 0.f ? (M + log2f(Z)) * kLn2 : -INFINITY;
            if (p.status && bh == 0) *p.status = MKA_OK;
        }
    }
    cluster_sync();
}

// GROUPS > 1: many chunks, dealt in turn to that many groups of DH threads (a thread per column each).
template <int DH, int GROUPS>
__global__ void __launch_bounds__(DH * GROUPS) decode_combine_kernel(const DecodeParams p) {
    chain_enter();
    constexpr int kThreads = DH * GROUPS;
    const long long bh = blockIdx.x;
    const int b = (int)(bh / p.H);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, col = tid % DH, grp = tid / DH;
    const float* part = p.partial + bh * p.total_chunks * (DH + 2);
    float lam[3] = {1.f, 1.f, 1.f};
    // The kernel is a chain of memory round trips, so all that may be needed is asked for at once, bounded by the room that there is: the
    // number of partials, the maxima and sums, and the accumulators of the first chunks.  (112 heads x 20 chunks: 8.6 us with three trips
    // one after the other, 6.3 with two.  28 heads x 56 chunks: 5.5 us with two and a third for the chunks past 32.)
    constexpr int kAhead = GROUPS == 1 ? 32 : 16;
    const int n_room = (int)(p.total_chunks - (p.counted ? 1 : 0));
    float count = 0.f;
    if (p.counted) {
        count = part[0];
        part += DH + 2;
    } else {
#pragma unroll
        for (int l = 0; l < 3; ++l) lam[l] = p.gate[b * 3 + l];
    }
    float m_own = -INFINITY, z_own = 0.f;                      // chunk tid's
    if (tid < n_room) { m_own = part[(long long)tid * (DH + 2)]; z_own = part[(long long)tid * (DH + 2) + 1]; }
    float ahead[kAhead];
#pragma unroll
    for (int j = 0; j < kAhead; ++j) ahead[j] = grp + j * GROUPS < n_room ? part[(long long)(grp + j * GROUPS) * (DH + 2) + 2 + col] : 0.f;
    // (a call whose waits ran out may not have written the count)
    const long long total = !p.counted ? p.total_chunks : (count > 0.f ? (long long)fminf(count, (float)n_room) : 0);
    const long long c1 = p.n_chunks[0], c2 = c1 + p.n_chunks[1];
    // global maximum over the chunks that count (gate > 0 and something summed): warp shuffles, then
    // one shared-memory hop across the CTA's warps
    float M = -INFINITY;
    for (long long c = tid; c < total; c += kThreads) {
        const float g = c < c1 ? lam[0] : (c < c2 ? lam[1] : lam[2]);
        const float mc = c == tid ? m_own : part[c * (DH + 2)], zc = c == tid ? z_own : part[c * (DH + 2) + 1];
        if (g > 0.f && zc > 0.f) M = fmaxf(M, mc);
    }
    M = warp_max(M);
    __shared__ float sm[kThreads / 32];
    if (lane == 0) sm[warp] = M;
    __syncthreads();
    M = sm[0];
#pragma unroll
    for (int w = 1; w < kThreads / 32; ++w) M = fmaxf(M, sm[w]);

    // Weights of a batch of kThreads chunks are worked out side by side (one chunk per thread) and parked in shared
    // memory; the accumulation over the batch then runs without a branch, its loads independent of each other.
    float Z = 0.f, A = 0.f;
    __shared__ float sw[kThreads];
    if (M > -INFINITY) {
        for (long long c0 = 0; c0 < total; c0 += kThreads) {
            const long long c = c0 + tid;
            float w = 0.f;
            if (c < total) {
                const float g = c < c1 ? lam[0] : (c < c2 ? lam[1] : lam[2]);
                const float mc = c0 == 0 ? m_own : part[c * (DH + 2)], zc = c0 == 0 ? z_own : part[c * (DH + 2) + 1];
                if (g > 0.f && zc > 0.f) { w = g * exp2f(mc - M); Z = fmaf(w, zc, Z); }
            }
            __syncthreads();                                   // the previous batch has been consumed
            sw[tid] = w;
            __syncthreads();
            const int nb = total - c0 < kThreads ? (int)(total - c0) : kThreads;
            const float* at = part + c0 * (DH + 2) + 2 + col;
            int j = grp;
            if (c0 == 0) {
#pragma unroll
                for (int u = 0; u < kAhead; ++u)
                    if (grp + u * GROUPS < nb) A = fmaf(sw[grp + u * GROUPS], ahead[u], A);
                j += kAhead * GROUPS;
            }
            for (; j + 7 * GROUPS < nb; j += 8 * GROUPS) {
                float v[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) v[u] = at[(long long)(j + u * GROUPS) * (DH + 2)];
#pragma unroll
                for (int u = 0; u < 8; ++u) A = fmaf(sw[j + u * GROUPS], v[u], A);
            }
            for (; j < nb; j += GROUPS) A = fmaf(sw[j], at[(long long)j * (DH + 2)], A);
        }
    }
    // Z: every thread holds the share of its own chunks
    Z = warp_sum(Z);
    __shared__ float sz[kThreads / 32], sa[GROUPS > 1 ? GROUPS - 1 : 1][DH];
    if (lane == 0) sz[warp] = Z;
    if (GROUPS > 1 && grp > 0) sa[grp - 1][col] = A;
    __syncthreads();
    if (grp > 0) return;
    Z = 0.f;
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) Z += sz[w];
#pragma unroll
    for (int g = 1; g < GROUPS; ++g) A += sa[g - 1][col];
    __nv_bfloat16* O = static_cast<__nv_bfloat16*>(p.O) + bh * DH;
    O[col] = __float2bfloat16_rn(Z > 0.f ? A / Z : 0.f);
    if (p.status && bh == 0 && tid == 0) *p.status = MKA_OK;
    if (p.LSE && tid == 0) p.LSE[bh] = Z > 0.f ? (M + log2f(Z)) * kLn2 : -INFINITY;
}

// Four groups where a thread would have many chunks and the CTAs leave SMs idle; at d = 64, where a group is two warps, for well more than it
// asks for at once.  Whole decode of grouped heads, four groups over one, lists of 1500 / 6500 / 20,000 rows, by the partials of a list of equal lengths:
//   d = 128   3 to 8 partials (160 to 288 heads)  0.98 .. 0.99 / 0.95 .. 0.99 / 0.97 .. 0.99      10  0.98 .. 1.05 / 0.94 .. 0.97 / 0.97 .. 0.99
//             19 and 25  0.99 .. 1.00 / 0.94 .. 0.95 / 0.95 .. 0.97      38 and 75  0.96 .. 0.99 / 0.87 .. 0.88 / 0.87 .. 0.92      297  1.05 / 0.86 / 0.63 .. 0.65
//   d = 64    up to 25  1.02 .. 1.08 / 1.01 .. 1.07 / 1.00 .. 1.04      38  1.06 .. 1.09 / 1.01 / 1.02      75  1.04 / 0.90 / 0.90      297  0.99 .. 1.04 / 0.79 .. 0.85 / 0.70
// (28 heads on 4 at 6500 rows, d = 128: 14.2 us, 12.4; a list of 1500 rows fills fewer partials than its share of the CTAs).  Chunks cut on the host: 34 and 40 of them 0.99 .. 1.00, 86 and
// 89 0.96 .. 1.00, 157 0.81 .. 0.91, 235 and more 0.55 .. 0.75.
template <int DH>
cudaError_t launch_combine(const DecodeParams& p, cudaStream_t st) {
    const dim3 grid((unsigned)((long long)p.B * p.H));
    if ((p.counted ? p.expected > (DH == 128 ? 2 : 48) : p.total_chunks > 32) && grid.x <= 296) return launch_chained(decode_combine_kernel<DH, 4>, grid, dim3(DH * 4), 0, st, 0, p);
    return launch_chained(decode_combine_kernel<DH, 1>, grid, dim3(DH), 0, st, 0, p);
}

// CTAs per (batch, head) of the one-kernel form, 0 = the split form.  As many as keep all clusters resident at once (296 CTAs);
// more only add rounds.  The split form's chunks fill the chip to the end, at 6.8 TB/s, and cost 10 us more (a second kernel, its
// launch, the partials).  A cluster's CTAs are as long as their pair's list: an SM brings its own at 52 GB/s, so SMs that hold two
// while others hold one finish last, and a last round with few CTAs leaves most of the chip idle.  Both are added up here; the
// model was fitted to 500 sizes of 8 to 2048 pairs and 200 to 16,000 rows, over which the form it picks takes 0.1 % more
// than the better one on average, 7 % at most.  Split form / clusters of 1 / 2 / 4 / 8 in us, chosen in brackets, d = 128:
//   8 pairs x 1000 rows    13.6 / 14.9 / 10.5 / 10.5 / [10.5]     128 x 10,000   113 / 168 / [109] / 113 / 123
//   96 x 5000     [49.4] / 85.9 / 54.4 / 59.2 / 53.5              288 x 5000     128 / [119] / 126 / 152
//   192 x 4000    [71.9] / 82.2 / 88.2 / 75.0                     304 x 2300     [69.8] / 93.1 / 78.4
//   304 x 4000    [111] / 152 / 127                               416 x 2300     [90.4] / 101 / 86.0
//   448 x 2300    [96.4] / 101 / 105                              640 x 3000     [166] / 194
int cluster_rule(const DecodeParams& p) {
    const long long rows = p.L[0].n + p.L[1].n + p.L[2].n, bh = (long long)p.B * p.H;
    int size = 1;
    while (size < kMaxCluster && bh * size * 2 <= 296) size *= 2;
    const long long ctas = bh * size;
    const double per_cta = (double)rows / size;
    if (ctas > 0x7fffffffLL || per_cta > 8192.0) return 0;                // (longer ones were not measured)
    const double kb = per_cta * 4.0 * p.d * 1e-3, sm = kb / 52.0, chip = kb / 6800.0;      // us: one CTA on an SM; its share of the chip's rate
    const double full = (double)(ctas / 296), rest = (double)(ctas % 296);
    double t = full * (2.0 * sm > 296.0 * chip ? 2.0 * sm : 296.0 * chip);
    const double alone = (rest > 148.0 || full > 0.0 ? 2.0 : 1.0) * sm;
    if (rest > 0.0) t += alone > rest * chip ? alone : rest * chip;
    return t <= (double)ctas * chip + 10.0 ? size : 0;
}

template <int DH>
cudaError_t launch_t(const DecodeParams& p, cudaStream_t st) {
    const long long bh = (long long)p.B * p.H;
    if (bh == 0) return cudaSuccess;
    if (const int size = cluster_rule(p))
        return launch_chained(decode_cluster_kernel<DH>, dim3((unsigned)(bh * size)), dim3(kWarps * 32), 0, st, size, p);
    if (p.total_chunks > 0) {
        cudaError_t e = launch_chained(decode_partial_kernel<DH>, dim3((unsigned)(bh * p.total_chunks)), dim3(kWarps * 32), 0, st, 0, p);
        if (e != cudaSuccess) return e;
    }
    return launch_combine<DH>(p, st);
}

}  // namespace

cudaError_t launch_decode_combine(const DecodeParams& p, cudaStream_t st) {
    const long long bh = (long long)p.B * p.H;
    if (bh == 0) return cudaSuccess;
    if (p.d != 128 && p.d != 64) return cudaErrorNotSupported;
    return p.d == 128 ? launch_combine<128>(p, st) : launch_combine<64>(p, st);
}

cudaError_t launch_decode(const DecodeParams& p, cudaStream_t st) {
    if (p.d == 128) return launch_t<128>(p, st);
    if (p.d == 64) return launch_t<64>(p, st);
    return cudaErrorNotSupported;
}

}  // namespace mka

// ---------------------------------------------------------------------------------------------
// mka_decode_static: the decode entry point for callers that cannot hand over scratch memory.
// The per-chunk partials live in the file-scope device array below instead of a caller workspace.
// Every GPU that loads this library carries the array (8 MiB) until the process exits.
namespace mka {
namespace {

constexpr size_t kStaticScratchFloats = (size_t)2 << 20;                    // 2 Mi floats = 8 MiB
static __device__ __align__(256) float g_decode_static_scratch[kStaticScratchFloats];

constexpr int kMaxDevices = 64;
float* g_static_scratch_ptr[kMaxDevices];       // device address of the array, per device ordinal
std::mutex g_static_scratch_mutex;

// In host code the array's name is only a handle; the address a kernel can use has to be asked for,
// once per device and with that device current.  With CUDA's lazy module loading that request (or the first
// launch from this file) is also the moment the 8 MiB are really taken on that device, so it can fail when the
// device has no memory left: the caller then sees MKA_ERR_CUDA from its first call.  The remembered address
// belongs to the device's current context and is not refreshed after a cudaDeviceReset.
cudaError_t static_scratch_address(float** out) {
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_static_scratch_mutex);
    if (!g_static_scratch_ptr[dev]) {
        float* ptr = nullptr;
        e = cudaGetSymbolAddress(reinterpret_cast<void**>(&ptr), g_decode_static_scratch);
        if (e != cudaSuccess) return e;
        if (!ptr) return cudaErrorInvalidSymbol;
        g_static_scratch_ptr[dev] = ptr;
    }
    *out = g_static_scratch_ptr[dev];
    return cudaSuccess;
}

inline bool is_aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

}  // namespace
}  // namespace mka

extern "C" size_t mka_decode_static_max_bytes(void) { return mka::kStaticScratchFloats * sizeof(float); }

extern "C" mka_status mka_decode_static(const mka_shape* s, const void* q, const mka_level L[3], const float* gate,
                                        void* O, float* LSE, void* stream) {
    using namespace mka;
    if (!s || !L) return MKA_ERR_ARG;
    if (s->dtype != MKA_BF16 || s->mode != MKA_MODE_FAST) return MKA_ERR_UNSUPPORTED;
    if (s->B < 0 || s->H < 0 || s->T != 1) return MKA_ERR_SHAPE;
    if (s->d != 64 && s->d != 128) return MKA_ERR_SHAPE;
    if (s->kv_heads < 0 || (s->kv_heads > 0 && (s->H % s->kv_heads != 0))) return MKA_ERR_SHAPE;
    int64_t n_level[3];
    for (int l = 0; l < 3; ++l) {
        n_level[l] = L[l].n;
        if (L[l].n < 0) return MKA_ERR_SHAPE;
        if (L[l].n == 0) continue;
        if (!L[l].k || !L[l].v) return MKA_ERR_ARG;
        if (L[l].stride_n < s->d || L[l].stride_b < 0 || L[l].stride_h < 0) return MKA_ERR_SHAPE;
        if (!is_aligned16(L[l].k) || !is_aligned16(L[l].v)) return MKA_ERR_ALIGN;
        if (L[l].stride_n % 8 || L[l].stride_b % 8 || L[l].stride_h % 8) return MKA_ERR_ALIGN;
    }
    if (s->B == 0 || s->H == 0) return MKA_OK;
    if (!q || !gate || !O) return MKA_ERR_ARG;
    if (!is_aligned16(q) || !is_aligned16(O)) return MKA_ERR_ALIGN;
    mka_decode_plan_t plan;
    mka_status st = mka_decode_plan(n_level, s->B, s->H, s->d, &plan);
    if (st != MKA_OK) return st;
    const unsigned long long slots = (unsigned long long)s->B * s->H * (unsigned long long)plan.total_chunks;
    if (slots > 0x7fffffffULL) return MKA_ERR_SHAPE;
    // the split table of this problem needs more partial slots than the built-in array holds
    if (slots * (unsigned long long)(s->d + 2) > kStaticScratchFloats) return MKA_ERR_WORKSPACE;
    float* scratch = nullptr;
    if (static_scratch_address(&scratch) != cudaSuccess) return MKA_ERR_CUDA;
    DecodeParams p = {};                 // (no partial counts, no status word)
    p.q = q; p.O = O; p.LSE = LSE; p.gate = gate;
    for (int l = 0; l < 3; ++l) {
        p.L[l].k = L[l].k; p.L[l].v = L[l].v; p.L[l].n = L[l].n;
        p.L[l].sb = L[l].stride_b; p.L[l].sh = L[l].stride_h; p.L[l].sn = L[l].stride_n;
        p.n_chunks[l] = plan.n_chunks[l];
    }
    p.B = s->B; p.H = s->H; p.d = s->d;
    p.kv_group = s->kv_heads > 0 ? s->H / s->kv_heads : 1;
    p.scale = s->scale > 0.f ? s->scale : 1.0f / sqrtf((float)s->d);
    p.chunk_rows = plan.chunk_rows;
    p.total_chunks = plan.total_chunks;
    // Nothing in the array has to start at zero: the partial kernel writes every slot that the combine
    // kernel of the same call reads, so whatever an earlier call left behind is never looked at.
    p.partial = scratch;
    cudaError_t e = launch_decode(p, static_cast<cudaStream_t>(stream));
    if (e == cudaErrorNotSupported) return MKA_ERR_UNSUPPORTED;
    return e == cudaSuccess ? MKA_OK : MKA_ERR_CUDA;
}

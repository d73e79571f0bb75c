// Router gate kernel: lambda = softmax over three levels of (R W_r + b_r), one gate per token
// (Alg. 1 step 12 / Alg. 2 step 5), plus the hard top-1 / top-2 and uniform routing variants
// (Table 10).  HBM-bound for many rows, latency-bound for few: every row of R is read exactly once with 16-byte loads.
// Also the router's backward: dW_r = R^T dG, db_r = sum dG (two deterministic passes).
#include <type_traits>

#include "common.cuh"

namespace mka {
namespace {

constexpr int kRowsPerWarp = 4;
constexpr int kWarps = 8;

__device__ __forceinline__ void finish_row(float g0, float g1, float g2, int route, long long row, float* gate,
                                           float* log2_gate, int8_t* idx) {
    float g[3] = {g0, g1, g2};
    float mx = fmaxf(g0, fmaxf(g1, g2));
    float e[3], sum = 0.f;
#pragma unroll
    for (int l = 0; l < 3; ++l) { e[l] = expf(g[l] - mx); sum += e[l]; }
    float lam[3];
#pragma unroll
    for (int l = 0; l < 3; ++l) lam[l] = e[l] / sum;
    int8_t id0 = -1, id1 = -1;
    if (route == MKA_ROUTE_UNIFORM) {
        lam[0] = lam[1] = lam[2] = 1.0f / 3.0f;
    } else if (route == MKA_ROUTE_TOP1 || route == MKA_ROUTE_TOP2) {
        int keep = route == MKA_ROUTE_TOP1 ? 1 : 2;
        bool kept[3] = {false, false, false};
        for (int k = 0; k < keep; ++k) {            // largest logit first; a tie goes to the lower level
            int best = -1;
#pragma unroll
            for (int l = 0; l < 3; ++l)
                if (!kept[l] && (best < 0 || g[l] > g[best])) best = l;
            kept[best] = true;
        }
        float ks = 0.f;
#pragma unroll
        for (int l = 0; l < 3; ++l) if (kept[l]) ks += lam[l];
#pragma unroll
        for (int l = 0; l < 3; ++l) lam[l] = kept[l] ? lam[l] / ks : 0.f;
#pragma unroll
        for (int l = 0; l < 3; ++l)
            if (kept[l]) { if (id0 < 0) id0 = (int8_t)l; else id1 = (int8_t)l; }
    }
#pragma unroll
    for (int l = 0; l < 3; ++l) {
        gate[row * 3 + l] = lam[l];
        if (log2_gate) log2_gate[row * 3 + l] = lam[l] > 0.f ? log2f(lam[l]) : -INFINITY;
    }
    if (idx) { idx[row * 2] = id0; idx[row * 2 + 1] = id1; }
}

template <typename T> struct Vec8;  // eight consecutive elements as floats
template <> struct Vec8<__nv_bfloat16> {
    using Raw = uint4;
    static __device__ __forceinline__ Raw fetch(const __nv_bfloat16* p) { return __ldg(reinterpret_cast<const uint4*>(p)); }
    static __device__ __forceinline__ void widen(const Raw& u, float (&x)[8]) {
        const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            x[2 * i] = __uint_as_float(w[i] << 16);
            x[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
        }
    }
};
template <> struct Vec8<float> {
    struct Raw { float4 a, b; };
    static __device__ __forceinline__ Raw fetch(const float* p) {
        return {__ldg(reinterpret_cast<const float4*>(p)), __ldg(reinterpret_cast<const float4*>(p) + 1)};
    }
    static __device__ __forceinline__ void widen(const Raw& u, float (&x)[8]) {
        x[0] = u.a.x; x[1] = u.a.y; x[2] = u.a.z; x[3] = u.a.w; x[4] = u.b.x; x[5] = u.b.y; x[6] = u.b.z; x[7] = u.b.w;
    }
};

template <typename T, int N> struct Cols : Vec8<T> {};   // N consecutive elements as floats
template <> struct Cols<__nv_bfloat16, 4> {
    using Raw = uint2;
    static __device__ __forceinline__ Raw fetch(const __nv_bfloat16* p) { return __ldg(reinterpret_cast<const uint2*>(p)); }
    static __device__ __forceinline__ void widen(const Raw& u, float (&x)[4]) {
        x[0] = __uint_as_float(u.x << 16); x[1] = __uint_as_float(u.x & 0xffff0000u);
        x[2] = __uint_as_float(u.y << 16); x[3] = __uint_as_float(u.y & 0xffff0000u);
    }
};
template <> struct Cols<float, 4> {
    using Raw = float4;
    static __device__ __forceinline__ Raw fetch(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }
    static __device__ __forceinline__ void widen(const Raw& u, float (&x)[4]) { x[0] = u.x; x[1] = u.y; x[2] = u.z; x[3] = u.w; }
};

// Sums of ROWS rows x 3 logits over a warp: while a lane holds several rows it hands half of them to its partner and adds
// the partner's other half, so that four rows cost 18 shuffles instead of 60.  The lanes of group `row` (32 / ROWS of
// them) end with that row's sums in acc[0..2].
template <int ROWS>
__device__ __forceinline__ void sum_rows(float (&acc)[ROWS * 3], int lane, int& row) {
    int held = ROWS, off = 16;
    row = 0;
#pragma unroll
    for (int n = ROWS; n > 1; n >>= 1) {
        const bool up = (lane & off) != 0;
#pragma unroll
        for (int i = 0; i < n / 2 * 3; ++i) {
            const float give = up ? acc[i] : acc[i + n / 2 * 3];
            const float got = __shfl_xor_sync(0xffffffffu, give, off);
            acc[i] = (up ? acc[i + n / 2 * 3] : acc[i]) + got;
        }
        held >>= 1;
        row += up ? held : 0;
        off >>= 1;
    }
    for (; off > 0; off >>= 1)
#pragma unroll
        for (int l = 0; l < 3; ++l) acc[l] += __shfl_xor_sync(0xffffffffu, acc[l], off);
}

// One CTA takes ROWS rows and spreads D over its THREADS threads (COLS columns each per pass), so that the loads of a row are
// independent of each other: ROWS of them are in flight, whatever the number of rows.  The kernel is bound by
// one load's latency: a warp that walks four rows by itself took 11 us for ONE row of D = 4096.  With thousands of rows
// the order turns round (see router_rows_kernel).  A thread's columns of W_r lie 12 COLS bytes from its neighbour's, so a 16-byte read by a warp
// touches 24 lines at eight columns and 12 at four, and all of W_r (48 KB at D = 4096) goes through each CTA's L1: with four columns and
// twice the threads one row of 4096 takes 2.30 us instead of 2.56, 512 rows of 3584 3.84 instead of 4.78.  Past one round
// of CTAs it is the rows' own loads that count, and with four columns they shrink to 8 bytes: eight and 256 threads there (2000 rows of 2048: 4.1 us against 5.9).
template <typename T, int ROWS, int COLS, int THREADS>
__global__ void __launch_bounds__(THREADS)
router_kernel(const T* __restrict__ R, const float* __restrict__ W_r, const float* __restrict__ b_r,
              long long rows, int D, int route, float* __restrict__ gate, float* __restrict__ log2_gate,
              int8_t* __restrict__ idx) {
    using V = Cols<T, COLS>;
    __shared__ float part[THREADS / 32][ROWS * 3];
    chain_enter();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long row0 = (long long)blockIdx.x * ROWS;
    const long long last = rows - 1 - row0;                       // a row past the end reads the last one again
    float acc[ROWS * 3];
#pragma unroll
    for (int i = 0; i < ROWS * 3; ++i) acc[i] = 0.f;
    const T* base = R + row0 * (long long)D;
    constexpr int kUnroll = ROWS == 2 ? 2 : 1;                // both passes of D = 4096 at once: 512 rows of 3584 3.84 us against 4.01; one row, four rows: nothing, or slower
#pragma unroll kUnroll
    for (int c = threadIdx.x * COLS; c < D; c += blockDim.x * COLS) {
        typename V::Raw x[ROWS];
#pragma unroll
        for (int r = 0; r < ROWS; ++r) x[r] = V::fetch(base + (r <= last ? r : last) * D + c);
        float w[3 * COLS];
        const float4* wp = reinterpret_cast<const float4*>(W_r + (long long)c * 3);
#pragma unroll
        for (int i = 0; i < 3 * COLS / 4; ++i) {
            const float4 v = __ldg(wp + i);
            w[4 * i] = v.x; w[4 * i + 1] = v.y; w[4 * i + 2] = v.z; w[4 * i + 3] = v.w;
        }
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
            float f[COLS];
            V::widen(x[r], f);
#pragma unroll
            for (int i = 0; i < COLS; ++i)
#pragma unroll
                for (int l = 0; l < 3; ++l) acc[r * 3 + l] = fmaf(f[i], w[3 * i + l], acc[r * 3 + l]);
        }
    }
    int row = 0;
    sum_rows<ROWS>(acc, lane, row);
    if ((lane & (32 / ROWS - 1)) == 0) {
#pragma unroll
        for (int l = 0; l < 3; ++l) part[warp][row * 3 + l] = acc[l];
    }
    __syncthreads();
    if (threadIdx.x < ROWS && row0 + threadIdx.x < rows) {
        float g[3] = {0.f, 0.f, 0.f};
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w)
#pragma unroll
            for (int l = 0; l < 3; ++l) g[l] += part[w][threadIdx.x * 3 + l];
        if (b_r) { g[0] += b_r[0]; g[1] += b_r[1]; g[2] += b_r[2]; }
        finish_row(g[0], g[1], g[2], route, row0 + threadIdx.x, gate, log2_gate, idx);
    }
}

// Many rows: a warp owns four of them and walks D by itself; one read of W_r serves the four, nothing waits for a CTA's
// slowest warp and no barrier follows.
template <typename T>
__global__ void __launch_bounds__(kWarps * 32)
router_rows_kernel(const T* __restrict__ R, const float* __restrict__ W_r, const float* __restrict__ b_r,
                   long long rows, int D, int route, float* __restrict__ gate, float* __restrict__ log2_gate,
                   int8_t* __restrict__ idx) {
    chain_enter();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long row0 = ((long long)blockIdx.x * kWarps + warp) * kRowsPerWarp;
    if (row0 >= rows) return;
    float acc[kRowsPerWarp * 3];
#pragma unroll
    for (int i = 0; i < kRowsPerWarp * 3; ++i) acc[i] = 0.f;
    const T* rp[kRowsPerWarp];
#pragma unroll
    for (int r = 0; r < kRowsPerWarp; ++r) rp[r] = R + (row0 + r < rows ? row0 + r : rows - 1) * (long long)D;   // a row past the end reads the last one again
    for (int c = lane * 8; c < D; c += 32 * 8) {
        float w[24];
        const float4* wp = reinterpret_cast<const float4*>(W_r + (long long)c * 3);
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            const float4 v = __ldg(wp + i);
            w[4 * i] = v.x; w[4 * i + 1] = v.y; w[4 * i + 2] = v.z; w[4 * i + 3] = v.w;
        }
#pragma unroll
        for (int r = 0; r < kRowsPerWarp; ++r) {
            float f[8];
            Vec8<T>::widen(Vec8<T>::fetch(rp[r] + c), f);
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int l = 0; l < 3; ++l) acc[r * 3 + l] = fmaf(f[i], w[3 * i + l], acc[r * 3 + l]);
        }
    }
    int row = 0;
    sum_rows<kRowsPerWarp>(acc, lane, row);
    if ((lane & (32 / kRowsPerWarp - 1)) == 0 && row0 + row < rows) {
        if (b_r) { acc[0] += b_r[0]; acc[1] += b_r[1]; acc[2] += b_r[2]; }
        finish_row(acc[0], acc[1], acc[2], route, row0 + row, gate, log2_gate, idx);
    }
}

// Any D and alignment: a warp walks four rows, one element a lane.
template <typename T>
__global__ void __launch_bounds__(kWarps * 32)
router_any_kernel(const T* __restrict__ R, const float* __restrict__ W_r, const float* __restrict__ b_r,
                  long long rows, int D, int route, float* __restrict__ gate, float* __restrict__ log2_gate,
                  int8_t* __restrict__ idx) {
    chain_enter();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long row0 = ((long long)blockIdx.x * kWarps + warp) * kRowsPerWarp;
    if (row0 >= rows) return;
    float acc[kRowsPerWarp][3];
#pragma unroll
    for (int r = 0; r < kRowsPerWarp; ++r) acc[r][0] = acc[r][1] = acc[r][2] = 0.f;
    const T* rp[kRowsPerWarp];
#pragma unroll
    for (int r = 0; r < kRowsPerWarp; ++r) {
        long long rr = row0 + r < rows ? row0 + r : rows - 1;   // clamp: tail rows recompute the last row
        rp[r] = R + rr * (long long)D;
    }
    for (int c = lane; c < D; c += 32) {
        float w0 = W_r[c * 3], w1 = W_r[c * 3 + 1], w2 = W_r[c * 3 + 2];
#pragma unroll
        for (int r = 0; r < kRowsPerWarp; ++r) {
            float x = Elem<T>::ld(rp[r] + c);
            acc[r][0] = fmaf(x, w0, acc[r][0]);
            acc[r][1] = fmaf(x, w1, acc[r][1]);
            acc[r][2] = fmaf(x, w2, acc[r][2]);
        }
    }
#pragma unroll
    for (int r = 0; r < kRowsPerWarp; ++r)
#pragma unroll
        for (int l = 0; l < 3; ++l) acc[r][l] = warp_sum(acc[r][l]);
    if (lane < kRowsPerWarp && row0 + lane < rows) {
        float g0 = 0.f, g1 = 0.f, g2 = 0.f;
#pragma unroll
        for (int r = 0; r < kRowsPerWarp; ++r)
            if (lane == r) { g0 = acc[r][0]; g1 = acc[r][1]; g2 = acc[r][2]; }
        if (b_r) { g0 += b_r[0]; g1 += b_r[1]; g2 += b_r[2]; }
        finish_row(g0, g1, g2, route, row0 + lane, gate, log2_gate, idx);
    }
}

// Sum of rows [r0, r1) of a [rows, 3] array by the 256 threads of a CTA, valid in thread 0.
template <typename V>
__device__ __forceinline__ void sum_dG(const V* __restrict__ x, long long r0, long long r1, double (&sm)[256][3], double (&a)[3]) {
    a[0] = a[1] = a[2] = 0.0;
    for (long long r = r0 + threadIdx.x; r < r1; r += 256)
#pragma unroll
        for (int l = 0; l < 3; ++l) a[l] += (double)x[r * 3 + l];
#pragma unroll
    for (int l = 0; l < 3; ++l) sm[threadIdx.x][l] = a[l];
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) {
        if (threadIdx.x < s)
#pragma unroll
            for (int l = 0; l < 3; ++l) sm[threadIdx.x][l] += sm[threadIdx.x + s][l];
        __syncthreads();
    }
#pragma unroll
    for (int l = 0; l < 3; ++l) a[l] = sm[0][l];
}

// The CTAs of the first column block also add up their chunk's rows of dG for db_r, in 64 bits because the rows' terms cancel
// (one CTA over all rows took 22 us at 32768 rows).
__device__ __forceinline__ void chunk_db(const float* __restrict__ dG, long long r0, long long r1, int chunk, double* __restrict__ db_partial) {
    if (blockIdx.x != 0 || !db_partial) return;
    __shared__ double sm[256][3];
    double b[3];
    sum_dG(dG, r0, r1, sm, b);
    if (threadIdx.x == 0)
#pragma unroll
        for (int l = 0; l < 3; ++l) db_partial[chunk * 3 + l] = b[l];
}

// dW_r partials: CTA (row chunk, column block); thread = one column of R, loops over the chunk's rows.
template <typename T>
__global__ void __launch_bounds__(256)
router_bwd_partial_kernel(const T* __restrict__ R, const float* __restrict__ dG, long long rows, int D,
                          int n_row_chunks, float* __restrict__ partial, double* __restrict__ db_partial) {
    chain_enter();
    const int c = blockIdx.x * 256 + threadIdx.x;
    const int chunk = blockIdx.y;
    const long long per = (rows + n_row_chunks - 1) / n_row_chunks;
    const long long r0 = chunk * per, r1 = r0 + per < rows ? r0 + per : rows;
    __shared__ float g[64][3];
    float a0 = 0.f, a1 = 0.f, a2 = 0.f;
    for (long long rb = r0; rb < r1; rb += 64) {
        __syncthreads();
        if (threadIdx.x < 64 * 3) {
            long long rr = rb + threadIdx.x / 3;
            g[threadIdx.x / 3][threadIdx.x % 3] = rr < r1 ? dG[rr * 3 + threadIdx.x % 3] : 0.f;
        }
        __syncthreads();
        if (c < D) {
            int lim = (int)((r1 - rb) < 64 ? (r1 - rb) : 64);
            for (int i = 0; i < lim; ++i) {
                float x = Elem<T>::ld(R + (rb + i) * (long long)D + c);
                a0 = fmaf(x, g[i][0], a0); a1 = fmaf(x, g[i][1], a1); a2 = fmaf(x, g[i][2], a2);
            }
        }
    }
    if (c < D) {
        float* o = partial + ((long long)chunk * D + c) * 3;
        o[0] = a0; o[1] = a1; o[2] = a2;
    }
    chunk_db(dG, r0, r1, chunk, db_partial);
}

// The same with N = 8 or 4 consecutive columns per lane (16- or 8-byte loads of bf16): a warp takes every eighth row of the chunk, and
// the next eight rows' loads are in flight while the current eight are added (without that the kernel waits for
// loads most of the time: 2 TB/s); the eight warps' sums meet in shared memory.  Used when D is a multiple of N and R is
// 16-byte aligned.
template <typename T, int N>
__global__ void __launch_bounds__(256, 2)
router_bwd_partial_vec_kernel(const T* __restrict__ R, const float* __restrict__ dG, long long rows, int D,
                           int n_row_chunks, float* __restrict__ partial, double* __restrict__ db_partial) {
    constexpr int kBatch = N * sizeof(T) <= 16 ? 8 : 4;        // rows of a batch: loads in flight a lane = 8
    __shared__ float sum[8][3 * N][33];
    chain_enter();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c = blockIdx.x * (32 * N) + lane * N;
    const int chunk = blockIdx.y;
    const long long per = (rows + n_row_chunks - 1) / n_row_chunks;
    const long long r0 = chunk * per, r1 = r0 + per < rows ? r0 + per : rows;
    float a[3 * N];
#pragma unroll
    for (int j = 0; j < 3 * N; ++j) a[j] = 0.f;
    typename Cols<T, N>::Raw x[2][kBatch];
    float g[2];
    // rows rb, rb + 8, ..; a row past the chunk's end reads row rb again and weighs 0.  Lane 3u + l fetches dG[row u][l].
    auto fetch = [&](long long rb, typename Cols<T, N>::Raw (&to)[kBatch], float& gv) {
        if (rb >= r1) return;
        if (c < D)
#pragma unroll
            for (int u = 0; u < kBatch; ++u) to[u] = Cols<T, N>::fetch(R + (rb + 8 * u < r1 ? rb + 8 * u : rb) * (long long)D + c);
        const long long gr = rb + 8 * (lane / 3);
        gv = lane < 3 * kBatch && gr < r1 ? __ldg(dG + gr * 3 + lane % 3) : 0.f;
    };
    auto add = [&](long long rb, const typename Cols<T, N>::Raw (&from)[kBatch], float gv) {
        if (rb >= r1) return;
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            const bool in = rb + 8 * u < r1;                   // (a repeated row weighs 0, but 0 x inf would not be 0)
            float f[N];
            Cols<T, N>::widen(from[u], f);
#pragma unroll
            for (int l = 0; l < 3; ++l) {
                const float gl = __shfl_sync(0xffffffffu, gv, 3 * u + l);
                if (in)
#pragma unroll
                    for (int j = 0; j < N; ++j) a[j * 3 + l] = fmaf(f[j], gl, a[j * 3 + l]);
            }
        }
    };
    fetch(r0 + warp, x[0], g[0]);
    for (long long rb = r0 + warp; rb < r1; rb += 16 * kBatch) {
        fetch(rb + 8 * kBatch, x[1], g[1]);
        add(rb, x[0], g[0]);
        fetch(rb + 16 * kBatch, x[0], g[0]);
        add(rb + 8 * kBatch, x[1], g[1]);
    }
#pragma unroll
    for (int j = 0; j < 3 * N; ++j) sum[warp][j][lane] = a[j];
    __syncthreads();
    const int cols = min(32 * N, D - (int)blockIdx.x * (32 * N)) * 3;
    for (int i = threadIdx.x; i < cols; i += 256) {
        float s = 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w) s += sum[w][i % (3 * N)][i / (3 * N)];
        partial[((long long)chunk * D + blockIdx.x * (32 * N)) * 3 + i] = s;
    }
    chunk_db(dG, r0, r1, chunk, db_partial);
}

// dW_r = sum of the chunks' partials (32 outputs to a CTA, eight threads to an output: the loads of one output are eight
// short chains, not one of 128); the last CTA instead gives db_r, from the chunks' sums or (db_partial null) from dG.
__global__ void __launch_bounds__(256) router_bwd_reduce_kernel(const float* __restrict__ partial, const float* __restrict__ dG, long long rows,
                                                                int D, int n_row_chunks, const double* __restrict__ db_partial,
                                                                float* __restrict__ dW_r, float* __restrict__ db_r) {
    chain_enter();
    if (db_r && blockIdx.x == gridDim.x - 1) {
        __shared__ double sm[256][3];
        double b[3];
        if (db_partial) sum_dG(db_partial, 0, n_row_chunks, sm, b);
        else sum_dG(dG, 0, rows, sm, b);
        if (threadIdx.x == 0)
#pragma unroll
            for (int l = 0; l < 3; ++l) db_r[l] = (float)b[l];
        return;
    }
    __shared__ float sm[8][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int i = blockIdx.x * 32 + lane;
    float s = 0.f;
    if (i < D * 3)
        for (int k = warp; k < n_row_chunks; k += 8) s += partial[(long long)k * D * 3 + i];
    sm[warp][lane] = s;
    __syncthreads();
    if (warp == 0 && i < D * 3) {
#pragma unroll
        for (int w = 1; w < 8; ++w) s += sm[w][lane];
        dW_r[i] = s;
    }
}

}  // namespace

namespace {
template <typename T>
cudaError_t router_t(const T* R, const float* W_r, const float* b_r, long long rows, int D, int route, float* gate, float* log2_gate,
              int8_t* idx, cudaStream_t st) {
    if (D % 8 || (uintptr_t)R % 16 || (uintptr_t)W_r % 16) {
        const long long rows_per_cta = kWarps * kRowsPerWarp;
        return launch_chained(router_any_kernel<T>, dim3((unsigned)((rows + rows_per_cta - 1) / rows_per_cta)), dim3(kWarps * 32), 0, st, 0,
                              R, W_r, b_r, rows, D, route, gate, log2_gate, idx);
    }
    // With many rows the warps have enough to do on their own, a row each, the sooner the shorter the rows are (us, a CTA's columns against the warps':
    // 9400 x 256 4.4, 3.7 and x 768 6.4, 6.0; 8192 x 1024 6.7, 7.5, 9400 x 1536 10.4, 10.1; 5000 x 4096 12.4, 20.7, 32768 x 2048 36, 28; loads ahead
    // of the sums and W_r in shared memory were slower too, 35 and 44).
    const int warps_from = D >= 2048 ? 64 : (D >= 1024 ? 56 : (D >= 768 ? 40 : 32));   // rows per SM
    if (rows >= warps_from * 148LL) {
        const long long rows_per_cta = kWarps * kRowsPerWarp;
        return launch_chained(router_rows_kernel<T>, dim3((unsigned)((rows + rows_per_cta - 1) / rows_per_cta)), dim3(kWarps * 32), 0, st, 0,
                              R, W_r, b_r, rows, D, route, gate, log2_gate, idx);
    }
    auto go = [&](auto kern, int per_cta, int cols, int most) {
        const int threads = D >= cols * most ? most : (D / cols + 31) / 32 * 32;
        return launch_chained(kern, dim3((unsigned)((rows + per_cta - 1) / per_cta)), dim3(threads), 0, st, 0, R, W_r, b_r, rows, D, route, gate,
                              log2_gate, idx);
    };
    // Below that D is spread over a CTA.  Few rows: one row to a CTA, then two, for the shortest chain, and four where their CTAs are enough (at 768 to
    // 2048 columns from two rows per SM on: 400 x 2048 with a forward behind it 17.0 us, four 16.6).  Then a launch lasts as long as its rounds of
    // resident CTAs: four columns a thread while all rows fit one, eight past it.  A CTA has a warp to 128 columns (four a thread, 16 at most) or to 256
    // (eight, 8 at most), and the registers let an SM hold 36 warps (fp32 32) of four rows by four columns, 32 of four by eight, 16 of eight by eight.
    // Routers one after the other, us, four by four / four by eight / eight by eight:
    //   1500 x 1024 bf16   [2.86] / 3.05 / 3.24     2000 x 1536 bf16   4.41 / [3.48] / 3.21     2500 x 512 fp32    [2.81] / 3.70 / 3.39
    //   2000 x 1024 bf16   [2.77] / 3.16 / 3.30     2000 x 4096 bf16   6.39 / [4.93] / 4.93     2500 x 4096 fp32   [8.42] / 10.3 / 10.2
    //   1500 x 1536 fp32     4.38 / 3.90 / [3.66]   3000 x 1024 fp32   4.32 / 4.24 / [3.90]     8192 x 3584 fp32   29.0 / [24.2] / 27.9
    // In bf16 a tensor-core forward follows, whose CTAs start beside the router's last ones if those leave them registers: eight rows by eight columns do not,
    // and behind them the pass is as long or longer (2626 x 1536: 40.9 us with four rows, 42.7 with eight, 2626 x 1024 35.2 and 35.7, 2000 x 1536 34.4 and 34.3).
    // Against one, two or eight rows by eight columns and warps from 32 rows per SM on, which was there before four columns a thread: 0.89 of the time over 16 widths from 128 to
    // 8192, 36 row counts and both types, routers one after the other; 12 of the 1152 sizes are slower by more than 4 %, by 9 % at most (2000 x 1536 bf16), none with
    // a forward behind it (50 sizes, 0.93).
    const bool fp32 = sizeof(T) == 4, mid = D >= 768 && D <= 2048;
    const int warps4 = D >= 16 * 128 ? 16 : (D + 127) / 128, warps8 = D >= 8 * 256 ? 8 : (D + 255) / 256;
    auto rounds = [&](int per_cta, int cta_warps, int sm_warps) {
        const long long per_round = 148LL * per_cta * (sm_warps / cta_warps);
        return (rows + per_round - 1) / per_round;
    };
    const long long n44 = rounds(4, warps4, fp32 ? 32 : 36), n48 = rounds(4, warps8, 32), n88 = rounds(8, warps8, 16);
    if (rows < 2 * 148) return go(router_kernel<T, 1, 4, 512>, 1, 4, 512);
    if (rows < 4 * 148 && !mid) return go(router_kernel<T, 2, 4, 512>, 2, 4, 512);
    // (short rows leave a CTA with two warps or less; long fp32 rows: three rounds of half the rows are shorter than two)
    const bool halves = fp32 && D > 2048 && n44 == 3 && (n48 < n88 ? n48 : n88) == 2;
    if ((n44 == 1 && (D > 256 || rows < 8 * 148)) || halves) return go(router_kernel<T, 4, 4, 512>, 4, 4, 512);
    if constexpr (sizeof(T) == 4) {                            // (a tie: eight rows read W_r half as often, four put more loads of R in flight)
        const bool tie8 = D <= 1024 || (n88 < 3 && (D <= 4096 || n88 == 1));
        if (D > 256 && (n88 < n48 || (n88 == n48 && tie8))) return go(router_kernel<T, 8, 8, 256>, 8, 8, 256);
    }
    return go(router_kernel<T, 4, 8, 256>, 4, 8, 256);
}
}  // namespace

cudaError_t launch_router(const void* R, const float* W_r, const float* b_r, long long rows, int D, int r_dtype,
                          int route, float* gate, float* log2_gate, int8_t* idx, cudaStream_t st) {
    if (rows == 0) return cudaSuccess;
    if (r_dtype == MKA_BF16) return router_t(static_cast<const __nv_bfloat16*>(R), W_r, b_r, rows, D, route, gate, log2_gate, idx, st);
    return router_t(static_cast<const float*>(R), W_r, b_r, rows, D, route, gate, log2_gate, idx, st);
}

cudaError_t launch_router_bwd(const void* R, int r_dtype, const float* dG, long long rows, int D, float* dW_r,
                              float* db_r, float* partial, double* db_partial, int n_row_chunks, cudaStream_t st) {
    // Columns a lane: eight where D and R allow it, else four, else one.  The vector kernels keep their own loads in flight and take
    // as many row chunks as fill the chip's CTA slots once (two to an SM).  A thread of the one-column kernel has one load in
    // flight and lives on the number of CTAs: it takes all of the caller's chunks.  Both kernels together, 32768 rows of bf16:
    // D = 4096 (eight columns) 69 us; D = 4100 87 us with four columns, 702 with one and few chunks; D = 2050 54 us with
    // all chunks, 397 with few; D = 4096 at an address that allows no vector 94 us, 697 with few.
    const bool aligned = (reinterpret_cast<uintptr_t>(R) & 15) == 0;
    const int cols = aligned && D % 8 == 0 ? 8 : (aligned && D % 4 == 0 ? 4 : 1);
    const int col_blocks = cols == 1 ? (D + 255) / 256 : (D + 32 * cols - 1) / (32 * cols);
    if (cols > 1 && n_row_chunks > 296 / col_blocks) n_row_chunks = 296 / col_blocks > 0 ? 296 / col_blocks : 1;
    double* db_part = dW_r && db_r ? db_partial : nullptr;
    cudaError_t e = cudaSuccess;
    if (dW_r) {
        const dim3 grid(col_blocks, n_row_chunks);
        auto launch = [&](const auto* r) {
            using T = std::remove_cv_t<std::remove_pointer_t<decltype(r)>>;
            auto kern = cols == 8 ? router_bwd_partial_vec_kernel<T, 8> : (cols == 4 ? router_bwd_partial_vec_kernel<T, 4> : router_bwd_partial_kernel<T>);
            e = launch_chained(kern, grid, dim3(256), 0, st, 0, r, dG, rows, D, n_row_chunks, partial, db_part);
        };
        if (r_dtype == MKA_BF16) launch(static_cast<const __nv_bfloat16*>(R));
        else launch(static_cast<const float*>(R));
    }
    const int blocks = (dW_r ? (D * 3 + 31) / 32 : 0) + (db_r ? 1 : 0);
    if (e != cudaSuccess || !blocks) return e;
    return launch_chained(router_bwd_reduce_kernel, dim3(blocks), dim3(256), 0, st, 0, partial, dG, rows, D, n_row_chunks, db_part, dW_r, db_r);
}

}  // namespace mka

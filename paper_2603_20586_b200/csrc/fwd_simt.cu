// CUDA-core forward of the gated three-level attention operator.
//   MKA_MODE_FAST: Eq. 5 -- exp(score) weighted by the level's gate, one running (max, sum, acc)
//                  state carried across all three levels (the max shift of Eq. 11-14, key blocks of
//                  32 rows as in Alg. 3, rescale of Eq. 13-14 applied on every block).
//   MKA_MODE_FULL: Alg. 1 -- one softmax state per level, outputs mixed by the gate at the end.
// fp32 arithmetic throughout, so this is the kernel for fp32 problems (tolerance 1e-4) and the
// on-GPU cross-check of the tensor-core kernel.  One CTA = 16 or 32 query rows of one (batch, head), see simt.cuh; a key tile of
// 32 rows is staged in shared memory as fp32 and each lane scores one key of the tile, four columns at a time.
#include <type_traits>

#include "simt.cuh"

namespace mka {
namespace {

template <typename T, int DH, int MODE, int GROUPS>
__global__ void __launch_bounds__(SimtCta<GROUPS>::kThreads, GROUPS == 1 ? 2 : 1) fwd_simt_kernel(const FwdParams p, const int vec) {
    chain_enter();
    using S = SimtCta<GROUPS>;
    constexpr int kRows = S::kRows, kGroupThreads = S::kWarps * 32;
    constexpr int NS = MODE == MKA_MODE_FULL ? 3 : 1;    // softmax states
    constexpr int CPL = DH / 32;                         // output columns per lane
    constexpr int LD = DH + 4, kTileFloats = kSimtTile * LD, R = kSimtWarpRows;
    extern __shared__ __align__(16) float smem[];
    float* qs = smem;                                    // [rows][DH]  tau * q
    float* ps = qs + kRows * DH;                         // [warps][4 rows][32]  weights of the warp's tile
    float* tiles = ps + S::kThreads * R;                 // [groups][K, V][32][LD]; at the end [groups][rows][NS][DH + 2]

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, group = warp / S::kWarps, wg = warp % S::kWarps, gtid = threadIdx.x % kGroupThreads;
    const int b = blockIdx.z, h = blockIdx.y;
    const long long t0 = (long long)blockIdx.x * kRows;
    const T* Q = static_cast<const T*>(p.Q) + (((long long)b * p.H + h) * p.T) * DH;
    T* O = static_cast<T*>(p.O) + (((long long)b * p.H + h) * p.T) * DH;

    if (p.status && threadIdx.x == 0 && (blockIdx.x | blockIdx.y | blockIdx.z) == 0) *p.status = MKA_OK;
    for (int i = threadIdx.x * 4; i < kRows * DH; i += S::kThreads * 4) {
        const long long t = t0 + i / DH;
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
        if (t < p.T) x = Fetch4<T>::at(Q + t * DH + i % DH, (vec & 8) != 0);
        qs[i] = x.x * p.scale; qs[i + 1] = x.y * p.scale; qs[i + 2] = x.z * p.scale; qs[i + 3] = x.w * p.scale;   // tau folded into q
    }
    float lam[3][R];
#pragma unroll
    for (int lvl = 0; lvl < 3; ++lvl)
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const long long t = t0 + wg * R + r, tc = t < p.T ? t : p.T - 1;
            lam[lvl][r] = p.gate[((long long)b * p.T + tc) * 3 + lvl];
        }

    float m[NS][R], z[NS][R], acc[NS][R][CPL];           // z: this lane's keys only
#pragma unroll
    for (int s = 0; s < NS; ++s)
#pragma unroll
        for (int r = 0; r < R; ++r) {
            m[s][r] = -INFINITY; z[s][r] = 0.f;
#pragma unroll
            for (int k = 0; k < CPL; ++k) acc[s][r][k] = 0.f;
        }

    float* ks = tiles + group * 2 * kTileFloats;
    float* vs = ks + kTileFloats;
    float* pw = ps + warp * R * 32;
    const float* qw = qs + wg * R * DH;
    const long long t_last = (t0 + kRows - 1 < p.T ? t0 + kRows - 1 : p.T - 1);
    int turns = 0;
    bool first = true;
#pragma unroll
    for (int lvl = 0; lvl < 3; ++lvl) {
        const int st = MODE == MKA_MODE_FULL ? lvl : 0;
        const LevelDev L = p.L[lvl];
        if (L.n == 0) continue;
        // union of the visible ranges of this CTA's rows
        long long lo_first, hi_first, lo_last, hi_last;
        visible_range(lvl, t0 + p.q_offset, p.window, L.n, p.decode, lo_first, hi_first);
        visible_range(lvl, t_last + p.q_offset, p.window, L.n, p.decode, lo_last, hi_last);
        const long long lo = lo_first, hi = hi_last > hi_first ? hi_last : hi_first;
        const T* Kp = static_cast<const T*>(L.k) + b * L.sb + (h / p.kv_group) * L.sh;
        const T* Vp = static_cast<const T*>(L.v) + b * L.sb + (h / p.kv_group) * L.sh;
        long long rlo[R], rhi[R];
        const long long j_first = lo / kSimtTile * kSimtTile;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const long long t = t0 + wg * R + r, tc = t < p.T ? t : p.T - 1;
            visible_range(lvl, tc + p.q_offset, p.window, L.n, p.decode, rlo[r], rhi[r]);
            if (t >= p.T) rhi[r] = rlo[r];
        }
        // the groups take the tiles of the three levels in turn, as one list
        int turn = group - turns % S::kGroups;
        if (turn < 0) turn += S::kGroups;
        if (hi > lo) turns += (int)((hi - j_first + kSimtTile - 1) / kSimtTile % S::kGroups);
        for (long long j0 = j_first + (long long)turn * kSimtTile; j0 < hi; j0 += S::kGroups * kSimtTile) {
            if (!first) group_sync<kGroupThreads>(group);               // the group's previous tile has been read
            load_pair<T, DH, kGroupThreads>(ks, vs, Kp, Vp, j0, L.n, L.sn, (vec >> lvl) & 1, gtid);
            copies_wait<T>();
            if (first) __syncthreads();                                 // the queries too
            else group_sync<kGroupThreads>(group);
            first = false;
            float s[R];
#pragma unroll
            for (int r = 0; r < R; ++r) s[r] = 0.f;
            const float* kr = ks + lane * LD;
#pragma unroll 4
            for (int c = 0; c < DH; c += 4) {
                const float4 kv = *reinterpret_cast<const float4*>(kr + c);
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const float4 q = *reinterpret_cast<const float4*>(qw + r * DH + c);
                    s[r] = fmaf(q.x, kv.x, s[r]); s[r] = fmaf(q.y, kv.y, s[r]); s[r] = fmaf(q.z, kv.z, s[r]); s[r] = fmaf(q.w, kv.w, s[r]);
                }
            }
            const long long j = j0 + lane;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const bool vis = (j >= rlo[r]) && (j < rhi[r]) && (MODE == MKA_MODE_FULL || lam[lvl][r] > 0.f);
                const float x = vis ? s[r] : -INFINITY;
                const float m_new = fmaxf(m[st][r], warp_max(x));
                float e = (m_new == -INFINITY) ? 0.f : expf(x - m_new);   // masked: exp(-inf) = 0
                const float resc = (m[st][r] == -INFINITY) ? 0.f : expf(m[st][r] - m_new);
                if (MODE == MKA_MODE_FAST) e *= lam[lvl][r];
                z[st][r] = z[st][r] * resc + e;
#pragma unroll
                for (int k = 0; k < CPL; ++k) acc[st][r][k] *= resc;
                m[st][r] = m_new;
                pw[r * 32 + lane] = e;
            }
            __syncwarp();
#pragma unroll 2
            for (int jj = 0; jj < kSimtTile; jj += 4) {
                float4 e[R];
#pragma unroll
                for (int r = 0; r < R; ++r) e[r] = *reinterpret_cast<const float4*>(pw + r * 32 + jj);
#pragma unroll
                for (int k = 0; k < CPL; ++k) {
                    const float* v = vs + jj * LD + lane + 32 * k;
                    const float v0 = v[0], v1 = v[LD], v2 = v[2 * LD], v3 = v[3 * LD];
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        acc[st][r][k] = fmaf(e[r].x, v0, acc[st][r][k]); acc[st][r][k] = fmaf(e[r].y, v1, acc[st][r][k]);
                        acc[st][r][k] = fmaf(e[r].z, v2, acc[st][r][k]); acc[st][r][k] = fmaf(e[r].w, v3, acc[st][r][k]);
                    }
                }
            }
            __syncwarp();
        }
    }

    // merge the groups: every group leaves (max, sum, acc) of its tiles, a warp then finishes one row after the other
    if (first) __syncthreads();                                         // a group without a tile
    __syncthreads();
    constexpr int kState = DH + 2;
#pragma unroll
    for (int s = 0; s < NS; ++s)
#pragma unroll
        for (int r = 0; r < R; ++r) {
            float* o = tiles + ((group * kRows + wg * R + r) * NS + s) * kState;
            const float zr = warp_sum(z[s][r]);
            if (lane == 0) { o[0] = m[s][r]; o[1] = zr; }
#pragma unroll
            for (int k = 0; k < CPL; ++k) o[2 + lane + 32 * k] = acc[s][r][k];
        }
    __syncthreads();
#pragma unroll 1
    for (int row = warp; row < kRows; row += S::kThreads / 32) {
    const long long t = t0 + row;
    if (t >= p.T) break;
    float out[CPL];
#pragma unroll
    for (int k = 0; k < CPL; ++k) out[k] = 0.f;
#pragma unroll
    for (int s = 0; s < NS; ++s) {
        const float* o = tiles + (row * NS + s) * kState;
        constexpr int kGroupFloats = kRows * NS * kState;
        // Eight groups' sums are added up in 64 bits, so that LSE is no further off than with the four groups of twice the rows (in 32 bits:
        // 0.6 to 1.8 % further on average over 30 inputs of six sizes, now 1.2 to 1.6 % nearer; fp32 step [1, 4, 256, 64] 81.5 us, now 81.7).
        std::conditional_t<S::kGroups == 8, double, float> sum = 0;
        float M = -INFINITY, A[CPL];
#pragma unroll
        for (int g = 0; g < S::kGroups; ++g) M = fmaxf(M, o[g * kGroupFloats]);
#pragma unroll
        for (int k = 0; k < CPL; ++k) A[k] = 0.f;
#pragma unroll
        for (int g = 0; g < S::kGroups; ++g) {
            const float mg = o[g * kGroupFloats], f = mg == -INFINITY ? 0.f : expf(mg - M);
            sum = fma(static_cast<decltype(sum)>(o[g * kGroupFloats + 1]), static_cast<decltype(sum)>(f), sum);
#pragma unroll
            for (int k = 0; k < CPL; ++k) A[k] = fmaf(o[g * kGroupFloats + 2 + lane + 32 * k], f, A[k]);
        }
        const float Z = static_cast<float>(sum);
        float w;
        if (MODE == MKA_MODE_FAST) {
            w = Z > 0.f ? 1.f / Z : 0.f;
            if (p.LSE && lane == 0) p.LSE[((long long)b * p.H + h) * p.T + t] = Z > 0.f ? M + logf(Z) : -INFINITY;
        } else {
            w = Z > 0.f ? p.gate[((long long)b * p.T + t) * 3 + s] / Z : 0.f;
        }
#pragma unroll
        for (int k = 0; k < CPL; ++k) out[k] = fmaf(A[k], w, out[k]);
    }
#pragma unroll
    for (int k = 0; k < CPL; ++k) Elem<T>::st(O + t * DH + lane + 32 * k, out[k]);
    }
}

template <typename T, int DH, int MODE, int GROUPS>
cudaError_t launch_g(const FwdParams& p, cudaStream_t st) {
    using S = SimtCta<GROUPS>;
    const dim3 grid((p.T + S::kRows - 1) / S::kRows, p.H, p.B);
    const size_t tiles = (size_t)S::kGroups * 2 * kSimtTile * (DH + 4), merge = (size_t)S::kGroups * S::kRows * (MODE == MKA_MODE_FULL ? 3 : 1) * (DH + 2);
    const size_t smem = sizeof(float) * (S::kRows * DH + S::kThreads * kSimtWarpRows + (tiles > merge ? tiles : merge));
    const int vec = simt_vec_bits(p.L, p.Q, nullptr, nullptr, sizeof(T) == 2 ? MKA_BF16 : MKA_F32);
    auto kern = fwd_simt_kernel<T, DH, MODE, GROUPS>;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return launch_chained(kern, grid, dim3(S::kThreads), smem, st, 0, p, vec);
}

template <typename T, int DH>
cudaError_t launch_t(const FwdParams& p, cudaStream_t st) {
    const int groups = simt_query_groups(p, 40.0);
    if constexpr (DH < 128) {                            // (eight groups' tiles of 128 columns do not fit shared memory)
        if (groups == 8) return p.mode == MKA_MODE_FULL ? launch_g<T, DH, MKA_MODE_FULL, 8>(p, st) : launch_g<T, DH, MKA_MODE_FAST, 8>(p, st);
    }
    if (p.mode == MKA_MODE_FULL) return groups == 4 ? launch_g<T, DH, MKA_MODE_FULL, 4>(p, st) : launch_g<T, DH, MKA_MODE_FULL, 1>(p, st);
    return groups == 4 ? launch_g<T, DH, MKA_MODE_FAST, 4>(p, st) : launch_g<T, DH, MKA_MODE_FAST, 1>(p, st);
}

template <typename T>
cudaError_t launch_d(const FwdParams& p, cudaStream_t st) {
    switch (p.d) {
        case 32: return launch_t<T, 32>(p, st);
        case 64: return launch_t<T, 64>(p, st);
        case 96: return launch_t<T, 96>(p, st);
        case 128: return launch_t<T, 128>(p, st);
        default: return cudaErrorNotSupported;
    }
}

}  // namespace

cudaError_t launch_fwd_simt(const FwdParams& p, int dtype, cudaStream_t st) {
    if (p.B == 0 || p.H == 0 || p.T == 0) return cudaSuccess;
    return dtype == MKA_BF16 ? launch_d<__nv_bfloat16>(p, st) : launch_d<float>(p, st);
}

}  // namespace mka

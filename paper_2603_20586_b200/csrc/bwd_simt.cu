// CUDA-core backward of Eq. 5 (derived by differentiating it; the paper prints no backward).
// With p = lambda exp(s - LSE) on the visible set, D_t = dO_t . O_t and dS = p (dO_t . v - D_t):
//   kernel dq    : dQ_t = tau sum_{l,j} dS k_{l,j};  per-head gate-logit gradient G[b,h,t,l] = sum_j dS;  D[b,h,t]
//   kernel dkv   : dK_{l,j} = tau sum_t dS q_t;  dV_{l,j} = sum_t p dO_t       (one launch for the three levels)
//   dG[b,t,l] = sum_h G[b,h,t,l] (fixed order): blocks of the dK/dV launch beside those of the key tiles
// Every output element is produced by exactly one CTA in a fixed summation order, so the result is
// deterministic.  fp32 arithmetic; 16 or 32 rows against tiles of 32, see simt.cuh.
#include <type_traits>

#include "simt.cuh"

namespace mka {
namespace {

template <typename T, int DH, int GROUPS>
__global__ void __launch_bounds__(SimtCta<GROUPS>::kThreads, GROUPS == 1 ? 2 : 1) bwd_dq_kernel(const BwdParams p, const int vec) {
    chain_enter();
    using S = SimtCta<GROUPS>;
    constexpr int kRows = S::kRows, kGroupThreads = S::kWarps * 32;
    constexpr int CPL = DH / 32, LD = DH + 4, kTileFloats = kSimtTile * LD, R = kSimtWarpRows;
    extern __shared__ __align__(16) float smem[];
    float* qs = smem;                            // [rows][DH]  tau * q
    float* gs = qs + kRows * DH;             // [rows][DH]  dO
    float* ps = gs + kRows * DH;                 // [warps][4 rows][32]  dS of the warp's tile
    float* tiles = ps + S::kThreads * R;         // [groups][K, V][32][LD]; at the end [groups][rows][DH + 6]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, group = warp / S::kWarps, wg = warp % S::kWarps, gtid = threadIdx.x % kGroupThreads;
    const int b = blockIdx.z, h = blockIdx.y;
    const long long t0 = (long long)blockIdx.x * kRows;
    const long long bh = (long long)b * p.H + h;
    const T* Q = static_cast<const T*>(p.Q) + bh * p.T * DH;
    const T* dO = static_cast<const T*>(p.dO) + bh * p.T * DH;
    if (threadIdx.x < 4 && (blockIdx.x | blockIdx.y | blockIdx.z) == 0) p.status[threadIdx.x] = 0u;
    for (int i = threadIdx.x * 4; i < kRows * DH; i += S::kThreads * 4) {
        const long long t = t0 + i / DH;
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f), y = x;
        if (t < p.T) {
            x = Fetch4<T>::at(Q + t * DH + i % DH, (vec & 8) != 0);
            y = Fetch4<T>::at(dO + t * DH + i % DH, (vec & 8) != 0);
        }
        qs[i] = x.x * p.scale; qs[i + 1] = x.y * p.scale; qs[i + 2] = x.z * p.scale; qs[i + 3] = x.w * p.scale;
        *reinterpret_cast<float4*>(gs + i) = y;
    }
    float lse[R], dlt[R], acc[R][CPL], lam[3][R], o_own[R][CPL];
    float Ap[R][3], Sp[R][3];                    // per level, this lane's keys: sum_j p dP and sum_j p (for the gate gradient)
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const long long t = t0 + wg * R + r, tc = t < p.T ? t : p.T - 1;
        lse[r] = p.LSE[bh * p.T + tc];
#pragma unroll
        for (int l = 0; l < 3; ++l) lam[l][r] = p.gate[((long long)b * p.T + tc) * 3 + l];
#pragma unroll
        for (int k = 0; k < CPL; ++k) {
            o_own[r][k] = Elem<T>::ld(static_cast<const T*>(p.O) + (bh * p.T + tc) * DH + lane + 32 * k);
            acc[r][k] = 0.f;
        }
        Ap[r][0] = Ap[r][1] = Ap[r][2] = 0.f;
        Sp[r][0] = Sp[r][1] = Sp[r][2] = 0.f;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < R; ++r) {
        // D_t = dO_t . O_t, left for the dK/dV kernel too
        const long long t = t0 + wg * R + r;
        float d = 0.f;
#pragma unroll
        for (int k = 0; k < CPL; ++k) d = fmaf(o_own[r][k], gs[(wg * R + r) * DH + lane + 32 * k], d);
        dlt[r] = warp_sum(d);
        if (group == 0 && lane == 0 && t < p.T) p.delta[bh * p.T + t] = dlt[r];
    }
    float* ks = tiles + group * 2 * kTileFloats;
    float* vs = ks + kTileFloats;
    float* pw = ps + warp * R * 32;
    const float* qw = qs + wg * R * DH;
    const float* gw = gs + wg * R * DH;
    const long long t_last = (t0 + kRows - 1 < p.T ? t0 + kRows - 1 : p.T - 1);
    int turns = 0;
#pragma unroll
    for (int lvl = 0; lvl < 3; ++lvl) {
        const LevelDev L = p.L[lvl];
        if (L.n == 0) continue;
        long long lo_f, hi_f, lo_l, hi_l;
        visible_range(lvl, t0 + p.q_offset, p.window, L.n, 0, lo_f, hi_f);
        visible_range(lvl, t_last + p.q_offset, p.window, L.n, 0, lo_l, hi_l);
        const long long lo = lo_f, hi = hi_l > hi_f ? hi_l : hi_f;
        const T* Kp = static_cast<const T*>(L.k) + b * L.sb + (h / p.kv_group) * L.sh;
        const T* Vp = static_cast<const T*>(L.v) + b * L.sb + (h / p.kv_group) * L.sh;
        long long rlo[R], rhi[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const long long t = t0 + wg * R + r, tc = t < p.T ? t : p.T - 1;
            visible_range(lvl, tc + p.q_offset, p.window, L.n, 0, rlo[r], rhi[r]);
            if (t >= p.T) rhi[r] = rlo[r];
        }
        // the groups take the tiles of the three levels in turn, as one list
        const long long j_first = lo / kSimtTile * kSimtTile;
        int turn = group - turns % S::kGroups;
        if (turn < 0) turn += S::kGroups;
        if (hi > lo) turns += (int)((hi - j_first + kSimtTile - 1) / kSimtTile % S::kGroups);
        for (long long j0 = j_first + (long long)turn * kSimtTile; j0 < hi; j0 += S::kGroups * kSimtTile) {
            group_sync<kGroupThreads>(group);
            load_pair<T, DH, kGroupThreads>(ks, vs, Kp, Vp, j0, L.n, L.sn, (vec >> lvl) & 1, gtid);
            copies_wait<T>();
            group_sync<kGroupThreads>(group);
            float s[R], dp[R];
#pragma unroll
            for (int r = 0; r < R; ++r) s[r] = dp[r] = 0.f;
            const float* kr = ks + lane * LD;
            const float* vr = vs + lane * LD;
#pragma unroll 2
            for (int c = 0; c < DH; c += 4) {
                const float4 kv = *reinterpret_cast<const float4*>(kr + c), vv = *reinterpret_cast<const float4*>(vr + c);
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const float4 q = *reinterpret_cast<const float4*>(qw + r * DH + c), g = *reinterpret_cast<const float4*>(gw + r * DH + c);
                    s[r] = fmaf(q.x, kv.x, s[r]); s[r] = fmaf(q.y, kv.y, s[r]); s[r] = fmaf(q.z, kv.z, s[r]); s[r] = fmaf(q.w, kv.w, s[r]);
                    dp[r] = fmaf(g.x, vv.x, dp[r]); dp[r] = fmaf(g.y, vv.y, dp[r]); dp[r] = fmaf(g.z, vv.z, dp[r]); dp[r] = fmaf(g.w, vv.w, dp[r]);
                }
            }
            const long long j = j0 + lane;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const bool vis = (j >= rlo[r]) && (j < rhi[r]) && lam[lvl][r] > 0.f;
                const float pr = vis ? lam[lvl][r] * expf(s[r] - lse[r]) : 0.f;
                pw[r * 32 + lane] = pr * (dp[r] - dlt[r]);
                Ap[r][lvl] = fmaf(pr, dp[r], Ap[r][lvl]);
                Sp[r][lvl] += pr;
            }
            __syncwarp();
#pragma unroll 2
            for (int jj = 0; jj < kSimtTile; jj += 4) {
                float4 e[R];
#pragma unroll
                for (int r = 0; r < R; ++r) e[r] = *reinterpret_cast<const float4*>(pw + r * 32 + jj);
#pragma unroll
                for (int k = 0; k < CPL; ++k) {
                    const float* v = ks + jj * LD + lane + 32 * k;
                    const float v0 = v[0], v1 = v[LD], v2 = v[2 * LD], v3 = v[3 * LD];
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        acc[r][k] = fmaf(e[r].x, v0, acc[r][k]); acc[r][k] = fmaf(e[r].y, v1, acc[r][k]);
                        acc[r][k] = fmaf(e[r].z, v2, acc[r][k]); acc[r][k] = fmaf(e[r].w, v3, acc[r][k]);
                    }
                }
            }
            __syncwarp();
        }
    }
    // merge the groups: a warp adds up one row after the other
    __syncthreads();
    constexpr int kState = DH + 6;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        float* o = tiles + (group * kRows + wg * R + r) * kState;
#pragma unroll
        for (int l = 0; l < 3; ++l) {
            const float a = warp_sum(Ap[r][l]), sp = warp_sum(Sp[r][l]);
            if (lane == 0) { o[l] = a; o[3 + l] = sp; }
        }
#pragma unroll
        for (int k = 0; k < CPL; ++k) o[6 + lane + 32 * k] = acc[r][k];
    }
    __syncthreads();
#pragma unroll 1
    for (int row = warp; row < kRows; row += S::kThreads / 32) {
    const long long t = t0 + row;
    if (t >= p.T) break;
    const float* o = tiles + row * kState;
    auto total = [&](int i) {
        float v = o[i];
#pragma unroll
        for (int g = 1; g < S::kGroups; ++g) v += o[g * kRows * kState + i];
        return v;
    };
    T* dQ = static_cast<T*>(p.dQ) + bh * p.T * DH;
#pragma unroll
    for (int k = 0; k < CPL; ++k) Elem<T>::st(dQ + t * DH + lane + 32 * k, total(6 + lane + 32 * k) * p.scale);
    // Gate-logit gradient G_l = sum_{j in l} p (dP - D).  Here D is taken as sum_{l,j} p dP / sum p, which
    // equals dO.O exactly in real arithmetic but does not inherit the rounding of O to its storage
    // type, so that sum_l G_l = 0 holds to fp32 accuracy.
    // (eight groups' sums in 64 bits, as in the forward)
    using Sum = std::conditional_t<S::kGroups == 8, double, float>;
    Sum a[3], sp[3];
#pragma unroll
    for (int l = 0; l < 3; ++l) {
        a[l] = o[l]; sp[l] = o[3 + l];
#pragma unroll
        for (int g = 1; g < S::kGroups; ++g) { a[l] += o[g * kRows * kState + l]; sp[l] += o[g * kRows * kState + 3 + l]; }
    }
    const Sum stot = sp[0] + sp[1] + sp[2];
    const Sum dd = stot > 0 ? (a[0] + a[1] + a[2]) / stot : 0;
#pragma unroll
    for (int l = 0; l < 3; ++l)
        if (lane == 0) p.Gpart[(bh * p.T + t) * 3 + l] = static_cast<float>(a[l] - sp[l] * dd);
    }
}

// One CTA = 16 or 32 key rows of one level of one (batch, KV head); its groups share the query tiles that see them.  One launch
// covers the three levels: blockIdx.x runs through L3's, L2's and L1's key tiles, the longest walks first, and then through the
// gate gradient's sums, which need nothing of dK and dV (with a launch of their own behind this one a step at [1, 4, 256, 64] took 91.9 us, now 85.9).
template <typename T, int DH, int GROUPS>
__global__ void __launch_bounds__(SimtCta<GROUPS>::kThreads, GROUPS == 1 ? 2 : 1) bwd_dkv_kernel(const BwdParams p, const int vec, const int key_tiles) {
    chain_enter();
    using S = SimtCta<GROUPS>;
    if (blockIdx.x >= (unsigned)key_tiles) {
        const long long at = ((long long)(blockIdx.x - key_tiles) * gridDim.y + blockIdx.y) * S::kThreads + threadIdx.x;
        if (at < p.T * 3LL) sum_dgate(p.Gpart, p.dG, p.H, p.T, blockIdx.z, at);
        return;
    }
    constexpr int kRows = S::kRows, kGroupThreads = S::kWarps * 32;
    constexpr int CPL = DH / 32, LD = DH + 4, kTileFloats = kSimtTile * LD, R = kSimtWarpRows;
    extern __shared__ __align__(16) float smem[];
    float* ksm = smem;                           // [rows][DH]  tau * k   (this CTA's key rows)
    float* vsm = ksm + kRows * DH;           // [rows][DH]
    float* ps = vsm + kRows * DH;                // [warps][p, dS][4 rows][32]
    float* tiles = ps + S::kThreads * 2 * R;     // [groups][Q, dO][32][LD]; at the end [groups][rows][2 DH]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, group = warp / S::kWarps, wg = warp % S::kWarps, gtid = threadIdx.x % kGroupThreads;
    const int b = blockIdx.z, h = blockIdx.y;               // h: KV head; its query heads h * G .. h * G + G - 1 are summed
    int lvl = 2;
    long long kt = blockIdx.x;
    while (kt >= (p.L[lvl].n + kRows - 1) / kRows) { kt -= (p.L[lvl].n + kRows - 1) / kRows; --lvl; }
    const LevelDev L = p.L[lvl];
    const LevelGradDev dL = p.dL[lvl];
    const long long j0 = kt * kRows;
    const T* Kp = static_cast<const T*>(L.k) + b * L.sb + h * L.sh;
    const T* Vp = static_cast<const T*>(L.v) + b * L.sb + h * L.sh;
    for (int i = threadIdx.x * 4; i < kRows * DH; i += S::kThreads * 4) {
        const long long j = j0 + i / DH;
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f), y = x;
        if (j < L.n) {
            x = Fetch4<T>::at(Kp + j * L.sn + i % DH, (vec >> lvl) & 1);
            y = Fetch4<T>::at(Vp + j * L.sn + i % DH, (vec >> lvl) & 1);
        }
        ksm[i] = x.x * p.scale; ksm[i + 1] = x.y * p.scale; ksm[i + 2] = x.z * p.scale; ksm[i + 3] = x.w * p.scale;
        *reinterpret_cast<float4*>(vsm + i) = y;
    }
    float accK[R][CPL], accV[R][CPL];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int k = 0; k < CPL; ++k) accK[r][k] = accV[r][k] = 0.f;
    // queries that can see any of this CTA's keys: positions p = t + q_offset with
    //   L1: j <= p <= j + W - 1   L2: p >= j   L3: all
    const long long j_last = (j0 + kRows - 1 < L.n ? j0 + kRows - 1 : L.n - 1);
    long long t_lo = 0, t_hi = p.T;
    if (lvl == 0) { t_lo = j0 - p.q_offset; t_hi = j_last + p.window - p.q_offset; }
    else if (lvl == 1) { t_lo = j0 - p.q_offset; }
    if (t_lo < 0) t_lo = 0;
    if (t_hi > p.T) t_hi = p.T;
    const long long first = t_lo / kSimtTile, per_head = t_hi > t_lo ? (t_hi + kSimtTile - 1) / kSimtTile - first : 0;
    float* qs = tiles + group * 2 * kTileFloats;
    float* gs = qs + kTileFloats;
    float* pw = ps + warp * 2 * R * 32;
    const float* kw = ksm + wg * R * DH;
    const float* vw = vsm + wg * R * DH;
    for (long long i = group; i < per_head * p.kv_group; i += S::kGroups) {     // head by head, each head's tiles in order
        const long long bh = (long long)b * p.H + (long long)h * p.kv_group + i / per_head;
        const long long tt = (first + i % per_head) * kSimtTile, t = tt + lane;   // lane = query of the tile; warp rows = keys
        const T* Q = static_cast<const T*>(p.Q) + bh * p.T * DH;
        const T* dO = static_cast<const T*>(p.dO) + bh * p.T * DH;
        const long long tc = t < p.T ? t : p.T - 1;
        const float lse = p.LSE[bh * p.T + tc], dlt = p.delta[bh * p.T + tc], lam = p.gate[((long long)b * p.T + tc) * 3 + lvl];
        if (i != group) group_sync<kGroupThreads>(group);
        load_pair<T, DH, kGroupThreads>(qs, gs, Q, dO, tt, p.T, DH, (vec & 8) != 0, gtid);
        copies_wait<T>();
        if (i == group) __syncthreads();                                        // the keys and values too
        else group_sync<kGroupThreads>(group);
        long long vlo, vhi;
        visible_range(lvl, t + p.q_offset, p.window, L.n, 0, vlo, vhi);
        if (t >= p.T) vhi = vlo;
        float s[R], dp[R];
#pragma unroll
        for (int r = 0; r < R; ++r) s[r] = dp[r] = 0.f;
        const float* qr = qs + lane * LD;
        const float* gr = gs + lane * LD;
#pragma unroll 2
        for (int c = 0; c < DH; c += 4) {
            const float4 qv = *reinterpret_cast<const float4*>(qr + c), gv = *reinterpret_cast<const float4*>(gr + c);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const float4 k = *reinterpret_cast<const float4*>(kw + r * DH + c), v = *reinterpret_cast<const float4*>(vw + r * DH + c);
                s[r] = fmaf(k.x, qv.x, s[r]); s[r] = fmaf(k.y, qv.y, s[r]); s[r] = fmaf(k.z, qv.z, s[r]); s[r] = fmaf(k.w, qv.w, s[r]);
                dp[r] = fmaf(v.x, gv.x, dp[r]); dp[r] = fmaf(v.y, gv.y, dp[r]); dp[r] = fmaf(v.z, gv.z, dp[r]); dp[r] = fmaf(v.w, gv.w, dp[r]);
            }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const long long j = j0 + wg * R + r;
            const bool vis = (j >= vlo) && (j < vhi) && lam > 0.f;
            const float pr = vis ? lam * expf(s[r] - lse) : 0.f;
            pw[r * 32 + lane] = pr;
            pw[(R + r) * 32 + lane] = pr * (dp[r] - dlt);
        }
        __syncwarp();
#pragma unroll 2
        for (int q = 0; q < kSimtTile; q += 4) {
            float4 pj[R], dj[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                pj[r] = *reinterpret_cast<const float4*>(pw + r * 32 + q);
                dj[r] = *reinterpret_cast<const float4*>(pw + (R + r) * 32 + q);
            }
#pragma unroll
            for (int k = 0; k < CPL; ++k) {
                const float* qc = qs + q * LD + lane + 32 * k;
                const float* gc = gs + q * LD + lane + 32 * k;
                const float q0 = qc[0], q1 = qc[LD], q2 = qc[2 * LD], q3 = qc[3 * LD];
                const float g0 = gc[0], g1 = gc[LD], g2 = gc[2 * LD], g3 = gc[3 * LD];
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    accK[r][k] = fmaf(dj[r].x, q0, accK[r][k]); accK[r][k] = fmaf(dj[r].y, q1, accK[r][k]);
                    accK[r][k] = fmaf(dj[r].z, q2, accK[r][k]); accK[r][k] = fmaf(dj[r].w, q3, accK[r][k]);
                    accV[r][k] = fmaf(pj[r].x, g0, accV[r][k]); accV[r][k] = fmaf(pj[r].y, g1, accV[r][k]);
                    accV[r][k] = fmaf(pj[r].z, g2, accV[r][k]); accV[r][k] = fmaf(pj[r].w, g3, accV[r][k]);
                }
            }
        }
        __syncwarp();
    }
    // merge the groups: a warp adds up one key row after the other
    if (group >= per_head * p.kv_group) __syncthreads();                        // a group without a tile
    __syncthreads();
#pragma unroll
    for (int r = 0; r < R; ++r) {
        float* o = tiles + (group * kRows + wg * R + r) * 2 * DH;
#pragma unroll
        for (int k = 0; k < CPL; ++k) { o[lane + 32 * k] = accK[r][k]; o[DH + lane + 32 * k] = accV[r][k]; }
    }
    __syncthreads();
#pragma unroll 1
    for (int row = warp; row < kRows; row += S::kThreads / 32) {
    const long long j = j0 + row;
    if (j >= L.n) break;
    const float* o = tiles + row * 2 * DH;
    T* dKp = static_cast<T*>(dL.dk) + b * dL.sb + h * dL.sh + j * dL.sn;
    T* dVp = static_cast<T*>(dL.dv) + b * dL.sb + h * dL.sh + j * dL.sn;
#pragma unroll
    for (int k = 0; k < CPL; ++k) {
        const int c = lane + 32 * k;
        float dk = o[c], dv = o[DH + c];
#pragma unroll
        for (int g = 1; g < S::kGroups; ++g) { dk += o[g * kRows * 2 * DH + c]; dv += o[g * kRows * 2 * DH + DH + c]; }
        Elem<T>::st(dKp + c, dk * p.scale);
        Elem<T>::st(dVp + c, dv);
    }
    }
}

// The gate gradient where the dK/dV launch cannot do it: no level has a key, dG is written over something that launch reads, or dQ comes after it.
__global__ void bwd_dgate_kernel(const float* Gpart, int B, int H, long long T, float* dG) {
    chain_enter();
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;   // over B*T*3
    if (i < (long long)B * T * 3) sum_dgate(Gpart, dG, H, T, i / (T * 3), i % (T * 3));
}

}  // namespace

cudaError_t launch_bwd_dgate(const float* Gpart, int B, int H, long long T, float* dG, cudaStream_t st) {
    const long long n = (long long)B * T * 3;
    if (n == 0) return cudaSuccess;
    return launch_chained(bwd_dgate_kernel, dim3((unsigned)((n + 255) / 256)), dim3(256), 0, st, 0, Gpart, B, H, T, dG);
}

namespace {

template <typename T, int DH, int GROUPS>
cudaError_t launch_dq(const BwdParams& p, int vec, cudaStream_t st) {
    using S = SimtCta<GROUPS>;
    const size_t smem = sizeof(float) * (2 * S::kRows * DH + S::kThreads * kSimtWarpRows + (size_t)S::kGroups * 2 * kSimtTile * (DH + 4));
    const cudaError_t e = cudaFuncSetAttribute(bwd_dq_kernel<T, DH, GROUPS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return launch_chained(bwd_dq_kernel<T, DH, GROUPS>, dim3((p.T + S::kRows - 1) / S::kRows, p.H, p.B), dim3(S::kThreads), smem, st, 0, p, vec);
}

template <typename T, int DH, int GROUPS>
cudaError_t launch_dkv(const BwdParams& p, int vec, cudaStream_t st) {
    using S = SimtCta<GROUPS>;
    long long key_tiles = 0;
    for (int l = 0; l < 3; ++l) key_tiles += (p.L[l].n + S::kRows - 1) / S::kRows;
    if (key_tiles == 0) return launch_bwd_dgate(p.Gpart, p.B, p.H, p.T, p.dG, st);
    const size_t smem = sizeof(float) * (2 * S::kRows * DH + S::kThreads * 2 * kSimtWarpRows + (size_t)S::kGroups * 2 * kSimtTile * (DH + 4));
    cudaError_t e = cudaFuncSetAttribute(bwd_dkv_kernel<T, DH, GROUPS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const int H_kv = p.H / (p.kv_group > 0 ? p.kv_group : 1);
    const long long gate_blocks = p.dg_last ? 0 : (p.T * 3LL + S::kThreads - 1) / S::kThreads;       // of a batch, dealt over blockIdx.x and .y
    e = launch_chained(bwd_dkv_kernel<T, DH, GROUPS>, dim3((unsigned)(key_tiles + (gate_blocks + H_kv - 1) / H_kv), H_kv, p.B), dim3(S::kThreads), smem, st, 0,
                       p, vec, (int)key_tiles);
    return e == cudaSuccess && p.dg_last ? launch_bwd_dgate(p.Gpart, p.B, p.H, p.T, p.dG, st) : e;
}

template <typename T, int DH>
cudaError_t launch_t(const BwdParams& p, cudaStream_t st) {
    const int vec = simt_vec_bits(p.L, p.Q, p.O, p.dO, sizeof(T) == 2 ? MKA_BF16 : MKA_F32);
    const int groups = simt_query_groups(p, 80.0);
    cudaError_t e;
    if constexpr (DH < 128) e = groups == 8 ? launch_dq<T, DH, 8>(p, vec, st) : (groups == 4 ? launch_dq<T, DH, 4>(p, vec, st) : launch_dq<T, DH, 1>(p, vec, st));
    else e = groups == 4 ? launch_dq<T, DH, 4>(p, vec, st) : launch_dq<T, DH, 1>(p, vec, st);
    if (e != cudaSuccess) return e;
    return simt_key_groups(p) ? launch_dkv<T, DH, 4>(p, vec, st) : launch_dkv<T, DH, 1>(p, vec, st);
}

template <typename T>
cudaError_t launch_d(const BwdParams& p, cudaStream_t st) {
    switch (p.d) {
        case 32: return launch_t<T, 32>(p, st);
        case 64: return launch_t<T, 64>(p, st);
        case 96: return launch_t<T, 96>(p, st);
        case 128: return launch_t<T, 128>(p, st);
        default: return cudaErrorNotSupported;
    }
}

}  // namespace

cudaError_t launch_bwd_simt(const BwdParams& p, int dtype, cudaStream_t st) {
    if (p.B == 0 || p.H == 0 || p.T == 0) return cudaSuccess;
    return dtype == MKA_BF16 ? launch_d<__nv_bfloat16>(p, st) : launch_d<float>(p, st);
}

}  // namespace mka

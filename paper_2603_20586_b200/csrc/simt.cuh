// Pieces shared by the CUDA-core forward and backward: tile loads and the shape of their CTAs.
// A CTA owns 16 rows (queries, or keys in the dK/dV kernel) and has four groups of four warps; every warp of a group owns
// four of the rows, and the groups take every fourth 32-row tile of the list that the rows walk, each into its own part
// of shared memory.  Their partial results are merged in a fixed order at the end.  Most problems that run here are small
// (fp32 reference runs: a few heads of a few hundred rows), so the launch is bound by the length of that walk on a
// mostly idle chip, not by arithmetic: with one group of eight warps over 32 rows, [1, 4, 256, 64] took 63 us.  Where the blocks
// fill the chip that one group of eight warps is the shape of the CTA (simt_four_groups).
#pragma once

#include "common.cuh"

namespace mka {

constexpr int kSimtTile = 32, kSimtWarpRows = 4;

// The shapes of a CTA, by its number of groups: eight groups of two warps (8 rows), four groups of four (16 rows), or one group of
// eight (32 rows).
template <int GROUPS> struct SimtCta {
    static constexpr int kGroups = GROUPS, kWarps = GROUPS == 8 ? 2 : (GROUPS == 4 ? 4 : 8);      // kWarps: of a group
    static constexpr int kRows = kWarps * kSimtWarpRows, kThreads = kGroups * kWarps * 32;
};

template <typename T> struct Fetch4;   // four consecutive elements as floats
template <> struct Fetch4<float> {
    static __device__ __forceinline__ float4 at(const float* p, bool vec) {
        if (vec) return __ldg(reinterpret_cast<const float4*>(p));
        return make_float4(__ldg(p), __ldg(p + 1), __ldg(p + 2), __ldg(p + 3));
    }
};
template <> struct Fetch4<__nv_bfloat16> {     // bf16 tensors are 16-byte aligned with strides that are multiples of 8
    static __device__ __forceinline__ float4 at(const __nv_bfloat16* p, bool) {
        const uint2 w = __ldg(reinterpret_cast<const uint2*>(p));
        return make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u), __uint_as_float(w.y << 16),
                           __uint_as_float(w.y & 0xffff0000u));
    }
};

// 32 rows [j0, j0 + 32) of two tensors of the same strides into shared memory, rows past n as zeros, by a group's threads.
// Pitch DH + 4 floats: rows stay 16-byte aligned and eight lanes' 16-byte reads of eight rows fall on different banks.
// All of a thread's pieces have to be on their way before the first one is waited for: a tile's 16 KB (d = 64, two warps) took 5300
// cycles when loads and stores to shared memory came in turn, of the 28,800 that the forward of [1, 4, 256, 64] lasted.  fp32 goes
// through asynchronous copies (the caller waits with copies_wait), bf16 through registers, which it has to be widened in anyway.  With the
// tiles of three levels dealt to the groups as one list (group 0 took the first tile of each level before) and gates and rows fetched
// with the first tile: forward 17.3 -> 14.6 us, backward 42.0 -> 38.4; [2, 8, 1024, 64] (window 500, 512 slots), all of it, 1996 -> 1818.
template <typename T, int DH, int GROUP_THREADS>
__device__ __forceinline__ void load_pair(float* da, float* db, const T* a, const T* b, long long j0, long long n, long long stride,
                                          bool vec, int gtid) {
    constexpr int V = DH / 4, N = kSimtTile * V / GROUP_THREADS;
    static_assert(N * GROUP_THREADS == kSimtTile * V, "a tile is dealt evenly");
    if constexpr (sizeof(T) == 4) {
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const int e = gtid + i * GROUP_THREADS, r = e / V, c = (e % V) * 4;
            const bool in = j0 + r < n;
            const long long at = in ? (j0 + r) * stride + c : 0;
            const uint32_t to_a = (uint32_t)__cvta_generic_to_shared(da + r * (DH + 4) + c), to_b = (uint32_t)__cvta_generic_to_shared(db + r * (DH + 4) + c);
            if (vec) {
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(to_a), "l"(a + at), "r"(in ? 16 : 0) : "memory");
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(to_b), "l"(b + at), "r"(in ? 16 : 0) : "memory");
            } else {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(to_a + 4 * k), "l"(a + at + (in ? k : 0)), "r"(in ? 4 : 0) : "memory");
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(to_b + 4 * k), "l"(b + at + (in ? k : 0)), "r"(in ? 4 : 0) : "memory");
                }
            }
        }
    } else {
        constexpr int kAhead = N <= 8 ? N : N / 2;           // pieces of each tensor in registers at a time
        static_assert(N % kAhead == 0, "the last turn would run past the tile");
#pragma unroll
        for (int i0 = 0; i0 < N; i0 += kAhead) {
            uint2 x[kAhead], y[kAhead];
#pragma unroll
            for (int i = 0; i < kAhead; ++i) {
                const int e = gtid + (i0 + i) * GROUP_THREADS, r = e / V, c = (e % V) * 4;
                x[i] = y[i] = make_uint2(0u, 0u);
                if (j0 + r < n) {
                    x[i] = __ldg(reinterpret_cast<const uint2*>(a + (j0 + r) * stride + c));
                    y[i] = __ldg(reinterpret_cast<const uint2*>(b + (j0 + r) * stride + c));
                }
            }
#pragma unroll
            for (int i = 0; i < kAhead; ++i) {
                const int e = gtid + (i0 + i) * GROUP_THREADS, r = e / V, c = (e % V) * 4;
                *reinterpret_cast<float4*>(da + r * (DH + 4) + c) = make_float4(__uint_as_float(x[i].x << 16), __uint_as_float(x[i].x & 0xffff0000u),
                                                                                __uint_as_float(x[i].y << 16), __uint_as_float(x[i].y & 0xffff0000u));
                *reinterpret_cast<float4*>(db + r * (DH + 4) + c) = make_float4(__uint_as_float(y[i].x << 16), __uint_as_float(y[i].x & 0xffff0000u),
                                                                                __uint_as_float(y[i].y << 16), __uint_as_float(y[i].y & 0xffff0000u));
            }
        }
    }
}
template <typename T> __device__ __forceinline__ void copies_wait() {
    if constexpr (sizeof(T) == 4) asm volatile("cp.async.wait_all;" ::: "memory");
}

template <int GROUP_THREADS>
__device__ __forceinline__ void group_sync(int group) { asm volatile("bar.sync %0, %1;" ::"r"(group + 1), "n"(GROUP_THREADS) : "memory"); }

// 16-byte loads are possible: bit l for level l (its K and V), bit 3 for the contiguous tensors.
inline int simt_vec_bits(const LevelDev L[3], const void* a, const void* b, const void* c, int dtype) {
    auto ok = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; };
    int bits = ok(a) && ok(b) && ok(c) ? 8 : 0;
    for (int l = 0; l < 3; ++l)
        if (ok(L[l].k) && ok(L[l].v) && L[l].sn % 4 == 0 && L[l].sh % 4 == 0 && L[l].sb % 4 == 0) bits |= 1 << l;
    return dtype == MKA_BF16 ? 15 : bits;
}

// Which shape.  Four groups shorten the walk of a CTA and leave fewer CTAs on an SM at a time: they are for launches whose blocks
// do not fill the chip, and for long walks; one group has the better throughput.  `blocks`: CTAs of 16 rows;
// `walk`: tiles that a row block visits, on average; `k`, tiles for a block more than one per SM: 40 in the forward,
// 80 for dQ and 120 (of the longest walk) for dK/dV, where four groups hold out longer.  Over 167 shapes of d = 32 to 128, timed with a tile's loads all in
// flight, the rule costs 1.6 % on average against the best shape in the forward at d = 32 and 64 (0.2 % above), 0.8 % (0.1) in the backward with dQ's,
// 0.2 % with dK/dV's; the most where a second round is nearly empty (the last of these).  fp32, us, four groups / one group:
//   forward, d = 64    [1, 8, 200], window 200, 300 slots, 104 blocks    29.1 / 63.4 (eight 31.9)    [3, 8, 200], 100 slots, 312    47.5 / 68.7
//                      [3, 8, 512], 100 slots, 768                       140 / 155                   [1, 8, 3000], 100 slots, 1504  718 / 777
//                      [1, 8, 1024], window 16, 32 slots, 512            108 / 132                   [8, 16, 64], 400 slots, 512    83.8 / 70.8
//   forward, d = 128   [4, 8, 200], window 100, 100 slots, 416           87.5 / 103
inline bool simt_four_groups(long long blocks, double walk, double k) { return blocks <= 148 || (double)(blocks - 148) <= k * walk; }
template <typename P> inline double simt_query_walk(const P& p) {                     // forward and dQ: row blocks of queries
    double keys = 0.0;
    for (int l = 0; l < 3; ++l) {
        const double n = (double)p.L[l].n, seen = l == 0 ? (double)p.window + 15.0 : (l == 1 ? (double)p.q_offset + 0.5 * p.T : n);
        keys += n > 0.0 ? 32.0 + (seen < n ? seen : n) : 0.0;
    }
    return keys / 32.0;
}
template <typename P> inline int simt_query_groups(const P& p, double k) {
    const long long blocks = (long long)p.B * p.H * ((p.T + 15) / 16);
    const double walk = simt_query_walk(p);
    // Half as many rows to a CTA where even twice the blocks find an SM each: a step of the walk takes as long (its sixteen warps wait at barriers and for
    // shared-memory reads, which are busy 22 to 35 % of the time) but covers eight tiles.  [1, 4, 256, 64] (window 64, 128 slots): both
    // forwards and the backward together 106 us in four groups, 94 in eight and with the longest key blocks of dK/dV first (clusters of
    // two to four CTAs of four groups instead: 118).  Walks of 5.5 to 8 tiles, four / eight: forward 9.1 / 7.4 (d = 32, 53 to 103 rows), 12.0 / 9.3 (d = 64,
    // 49 to 84), 15.1 / 11.6 (d = 96, 94); before a tile's loads were in flight together they were equal there.
    if (p.d < 128 && blocks * 2 <= 148 && walk >= 5.0) return 8;
    return simt_four_groups(blocks, walk, k) ? 4 : 1;
}
// dK/dV: the levels' key blocks walk very different numbers of query tiles, and a launch lasts at least as long as its longest walk
// (a long-term level of 64 rows under 8192 queries beside a window of 16: 603 / 1434 us), so that walk counts here, also against
// the launch's total over the CTA slots.
inline bool simt_key_groups(const BwdParams& p) {
    double longest = 0.0, total = 0.0;
    long long blocks = 0;
    for (int l = 0; l < 3; ++l) {
        if (p.L[l].n == 0) continue;
        const double seen = l == 0 && p.window + 15.0 < p.T ? p.window + 15.0 : (double)p.T;
        const double walk = seen * p.kv_group / 32.0;
        const long long n = (long long)p.B * (p.H / p.kv_group) * ((p.L[l].n + 15) / 16);
        longest = walk > longest ? walk : longest;
        total += (l == 1 ? 0.5 : 1.0) * walk * (double)n;
        blocks += n;
    }
    return simt_four_groups(blocks, longest, 120.0) || longest * 444.0 >= total;
}

}  // namespace mka

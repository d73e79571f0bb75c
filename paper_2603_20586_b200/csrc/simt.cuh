// Pieces shared by the CUDA-core forward and backward: tile loads and the shape of their CTAs.
// A CTA owns 16 rows (queries, or keys in the dK/dV kernel) and has four groups of four warps; every warp of a group owns
// four of the rows, and the groups take every fourth 32-row tile of the list that the rows walk, each into its own part
// of shared memory.  Their partial results are merged in a fixed order at the end.  The problems that run here are small
// (fp32 reference runs: a few heads of a few hundred rows), so the launch is bound by the length of that walk on a
// mostly idle chip, not by arithmetic: with one group of eight warps over 32 rows, [1, 4, 256, 64] took 63 us.
#pragma once

#include "common.cuh"

namespace mka {

constexpr int kSimtRows = 16, kSimtTile = 32, kSimtWarpRows = 4, kSimtGroups = 4, kSimtThreads = 512;

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

// 32 rows [j0, j0 + 32) of two tensors of the same strides into shared memory, rows past n as zeros, by a group's 128 threads.
// Pitch DH + 4 floats: rows stay 16-byte aligned and eight lanes' 16-byte reads of eight rows fall on different banks.
template <typename T, int DH>
__device__ __forceinline__ void load_pair(float* da, float* db, const T* a, const T* b, long long j0, long long n, long long stride,
                                          bool vec, int gtid) {
    constexpr int V = DH / 4;
#pragma unroll
    for (int i = 0; i < kSimtTile * V / 128; ++i) {
        const int e = gtid + i * 128, r = e / V, c = (e % V) * 4;
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f), y = x;
        if (j0 + r < n) {
            x = Fetch4<T>::at(a + (j0 + r) * stride + c, vec);
            y = Fetch4<T>::at(b + (j0 + r) * stride + c, vec);
        }
        *reinterpret_cast<float4*>(da + r * (DH + 4) + c) = x;
        *reinterpret_cast<float4*>(db + r * (DH + 4) + c) = y;
    }
}

__device__ __forceinline__ void group_sync(int group) { asm volatile("bar.sync %0, 128;" ::"r"(group + 1) : "memory"); }

// 16-byte loads are possible: bit l for level l (its K and V), bit 3 for the contiguous tensors.
inline int simt_vec_bits(const LevelDev L[3], const void* a, const void* b, const void* c, int dtype) {
    auto ok = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; };
    int bits = ok(a) && ok(b) && ok(c) ? 8 : 0;
    for (int l = 0; l < 3; ++l)
        if (ok(L[l].k) && ok(L[l].v) && L[l].sn % 4 == 0 && L[l].sh % 4 == 0 && L[l].sb % 4 == 0) bits |= 1 << l;
    return dtype == MKA_BF16 ? 15 : bits;
}

}  // namespace mka

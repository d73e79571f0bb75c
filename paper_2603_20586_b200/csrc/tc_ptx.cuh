// PTX wrappers shared by the tensor-core kernels (sm_100a): mbarrier, TMA tensor loads, tcgen05 matrix
// products with TMEM accumulators, TMEM loads/stores, and the shared-memory matrix descriptors for the
// 128-byte-swizzled panels that the TMA loads produce.  Internal header, not part of the C ABI.
#pragma once

#include <cuda.h>

#include "common.cuh"

namespace mka {

// Every device-side wait gives up after a wall-clock limit: one second unless mka_set_wait_limit_us changed it.
// The launchers read the limit on the host (wait_limit_ns) and pass it to the kernel, which keeps it in shared memory
// beside the flag that tells the other roles of the CTA that somebody gave up.
struct WaitCtl {
    int abort;                       // set by the first wait that ran out; every other wait of the CTA then returns false
    unsigned long long limit_ns;
};
unsigned long long wait_limit_ns();   // host

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint64_t* b, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* b, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(b)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* b) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(b)) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t* b, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
                 : "=r"(ok) : "r"(smem_u32(b)), "r"(parity) : "memory");
    return ok != 0;
}
__device__ __forceinline__ unsigned long long gtimer() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// Bounded wait: false when the limit (`limits` of them) expired or another role already gave up.
__device__ __forceinline__ bool mbar_wait(uint64_t* b, uint32_t parity, volatile WaitCtl* ctl, unsigned int limits = 1) {
    if (mbar_try(b, parity)) return true;
    const unsigned long long t0 = gtimer();
    for (;;) {
#pragma unroll 1
        for (int i = 0; i < 32; ++i)
            if (mbar_try(b, parity)) return true;
        if (ctl->abort) return false;
        if (gtimer() - t0 > limits * ctl->limit_ns) { ctl->abort = 1; return false; }
    }
}
// Waits for a copy that was issued.  Unlike mbar_wait it goes on when another role gave up: a CTA must not hand its shared memory
// back with a copy in flight.  Bounded by the same limit, counted from `t0`, so that several of these in a row have one limit.
__device__ __forceinline__ void mbar_drain(uint64_t* b, uint32_t parity, volatile WaitCtl* ctl, unsigned long long t0) {
    while (!mbar_try(b, parity))
        if (gtimer() - t0 > ctl->limit_ns) { ctl->abort = 1; return; }
}
__device__ __forceinline__ void tma_load_4d(void* dst, const CUtensorMap* map, int x, int y, int z, int w, uint64_t* bar) {
    asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
                 ::"r"(smem_u32(dst)), "l"(map), "r"(x), "r"(y), "r"(z), "r"(w), "r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, int x, int y, int z, uint64_t* bar) {
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
                 ::"r"(smem_u32(dst)), "l"(map), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar)) : "memory");
}
// Shared-memory matrix descriptors (128-byte swizzle; 8-row groups 1024 bytes apart).
__device__ __forceinline__ uint64_t desc_kmajor(uint32_t addr) {
    return (uint64_t)((addr >> 4) & 0x3FFF) | (1ull << 16) | (64ull << 32) | (1ull << 46) | (2ull << 61);
}
__device__ __forceinline__ uint64_t desc_mnmajor(uint32_t addr, uint32_t panel_stride_bytes) {
    return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)((panel_stride_bytes >> 4) & 0x3FFF) << 16) | (64ull << 32) |
           (1ull << 46) | (2ull << 61);
}
__device__ __forceinline__ void mma_ss(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
    asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}"
                 ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void mma_ts(uint32_t d, uint32_t a_tmem, uint64_t b, uint32_t idesc, uint32_t accumulate) {
    asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}"
                 ::"r"(d), "r"(a_tmem), "l"(b), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// The same descriptors split into their two 32-bit words.  The high word is one constant for every operand of
// these kernels; the low word is the start-address field (address >> 4: shared memory is smaller than 256 KB,
// so the 14-bit field cannot overflow and byte offsets are simply added as offset >> 4; in a cluster the
// address of a CTA's own shared memory carries its rank in higher bits, which are masked off)
// plus the leading-dimension field.  The issuing warp then spends one add per operand and matrix product.
constexpr uint32_t kDescHi = 64u | (1u << 14) | (2u << 29);
__device__ __forceinline__ uint32_t desc_lo_kmajor(uint32_t addr) { return ((addr >> 4) & 0x3FFF) | (1u << 16); }
__device__ __forceinline__ uint32_t desc_lo_mnmajor(uint32_t addr, uint32_t panel_stride_bytes) {
    return ((addr >> 4) & 0x3FFF) | ((panel_stride_bytes >> 4) << 16);
}
// Descriptor words of a K-major operand slab WITHOUT swizzle, 16 columns (one K-step) wide: core matrices of 8 rows x 16
// bytes; the two core matrices of a row group lie 128 bytes apart (leading-dimension field), row groups 256 bytes apart.
constexpr uint32_t kDescHiFlat = (256u >> 4) | (1u << 14);
__device__ __forceinline__ uint32_t desc_lo_flat(uint32_t addr) { return ((addr >> 4) & 0x3FFF) | ((128u >> 4) << 16); }
__device__ __forceinline__ uint64_t make_desc_flat(uint32_t lo) {
    uint64_t d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(lo), "r"(kDescHiFlat));
    return d;
}
__device__ __forceinline__ uint64_t make_desc(uint32_t lo) {
    uint64_t d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(lo), "r"(kDescHi));
    return d;
}
// offset (in descriptor units of 16 bytes) of K-step k inside a K-major tile whose 64-column panels are `panel` bytes apart
__device__ __forceinline__ constexpr uint32_t kstep_off(int k, uint32_t panel) {
    return ((uint32_t)(k / 4) * panel + (uint32_t)(k % 4) * 32u) >> 4;
}
// The matrix-product and commit instructions for a warp that runs its issue loop CONVERGED: every lane executes
// the block and elect.sync picks the one lane that issues.  Kept converged, the compiler can hold descriptors
// and addresses in uniform registers; issued from inside an `if (lane == 0)` region every operand has to be
// moved there first, which was measured at about 70 cycles per instruction -- more than the 64 cycles a
// 128x128x16 product takes to execute -- against at most 34 cycles this way.
__device__ __forceinline__ void mma_ss_elect(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
    asm volatile("{\n.reg .pred p, q;\nelect.sync _|q, 0xffffffff;\nsetp.ne.b32 p, %4, 0;\n@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}"
                 ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void mma_ts_elect(uint32_t d, uint32_t a_tmem, uint64_t b, uint32_t idesc, uint32_t accumulate) {
    asm volatile("{\n.reg .pred p, q;\nelect.sync _|q, 0xffffffff;\nsetp.ne.b32 p, %4, 0;\n@q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}"
                 ::"r"(d), "r"(a_tmem), "l"(b), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void mma_commit_elect(uint64_t* bar) {
    asm volatile("{\n.reg .pred q;\nelect.sync _|q, 0xffffffff;\n@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}"
                 ::"r"(smem_u32(bar)) : "memory");
}
// Bounded wait executed by every lane of a converged warp; the result is made warp-uniform.
__device__ __forceinline__ bool mbar_wait_warp(uint64_t* b, uint32_t parity, volatile WaitCtl* ctl, unsigned int limits = 1) {
    return __all_sync(0xffffffffu, mbar_wait(b, parity, ctl, limits));
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t* r) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
                   "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
                   "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]),
                   "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                 : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t* r) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
                   "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t* r) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};"
                 ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
                   "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]),
                   "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]),
                   "r"(r[30]), "r"(r[31]) : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t* r) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
                 ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
                   "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]) : "memory");
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t* r) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
                 ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]) : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// Packed pairs of fp32 (sm_100): one instruction works on two values held in an aligned register pair.
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(uint64_t r, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(r)); }
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
// 2^x for two arguments on the FMA pipe, for -126 <= x < 128 as good as ex2 (largest relative error 1.7e-7, that of ex2.approx is 2^-22): range reduction by rounding
// and a minimax polynomial.  x is clamped to -127 and split into n = round(x) and f = x - n in [-1/2, 1/2] by adding and subtracting
// 1.5 * 2^23 (the sum's low mantissa bits are n); 2^f is a polynomial of degree 5 with constant term exactly 1, fitted for the smallest maximum
// relative error (9.1e-8); n is added to the exponent field.  From -126 down to -127 that field is 0 and the result a subnormal number below the true one
// (ex2 gives 0 there); x <= -127 gives exactly 0, as ex2 does for -inf.  NaN gives 0 too: a caller whose arguments may be NaN has to
// see that by itself (fwd_tc_kernel's row maximum does).
__device__ __forceinline__ void exp2_pair_poly(float x0, float x1, float& p0, float& p1) {
    const float kMagic = 12582912.f;
    const uint64_t x = pack2(fmaxf(x0, -127.f), fmaxf(x1, -127.f));
    const uint64_t t = add2(x, pack2(kMagic, kMagic));
    const uint64_t n = add2(t, pack2(-kMagic, -kMagic));
    const uint64_t f = fma2(n, pack2(-1.f, -1.f), x);
    uint64_t r = fma2(pack2(0.0013264727f, 0.0013264727f), f, pack2(0.009671513f, 0.009671513f));
    r = fma2(r, f, pack2(0.055507336f, 0.055507336f));
    r = fma2(r, f, pack2(0.24022242f, 0.24022242f));
    r = fma2(r, f, pack2(0.693147f, 0.693147f));
    r = fma2(r, f, pack2(1.f, 1.f));
    float r0, r1, t0, t1;
    unpack2(r, r0, r1);
    unpack2(t, t0, t1);
    p0 = __uint_as_float(__float_as_uint(r0) + (__float_as_uint(t0) << 23));
    p1 = __uint_as_float(__float_as_uint(r1) + (__float_as_uint(t1) << 23));
}
// The largest of three; NaN if one of them is.
__device__ __forceinline__ float max3_nan(float a, float b, float c) {
    float d;
    asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
// Value at shared-memory address `addr` (of this CTA's layout) in CTA `rank` of the cluster.
__device__ __forceinline__ float ld_cluster(uint32_t addr, int rank) {
    uint32_t remote;
    float v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(addr), "r"(rank));
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(remote) : "memory");
    return v;
}
__device__ __forceinline__ float4 ld_cluster4(uint32_t addr, int rank) {
    uint32_t remote;
    float4 v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(addr), "r"(rank));
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(remote) : "memory");
    return v;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;" ::: "memory");
}
// The n lowest bits, 0 <= n <= 32 after clamping.
__device__ __forceinline__ uint32_t low_bits(int n) {
    n = max(0, min(n, 32));
    return (uint32_t)((1ull << n) - 1ull);
}
// x[l] with l known only at run time, without giving the array an address (it would live in local memory).
template <typename T> __device__ __forceinline__ T pick3(const T (&x)[3], int l) { return l == 0 ? x[0] : (l == 1 ? x[1] : x[2]); }
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

// Stores N = 16 or 32 consecutive columns of the warp's 32 rows (thread = row) as bf16.  A thread's own 16-byte pieces lie a
// row apart from its neighbours', so stored as they are every instruction touches 32 lines and the store unit takes one
// cycle for each; the lanes of a group first exchange pieces so that the group writes one row's N * 2 bytes at a
// time.  `row0` points at the first column of the warp's first row, `rows` of which (at most 32) exist.
template <int N>
__device__ __forceinline__ void store_rows_bf16(__nv_bfloat16* row0, long long stride, int rows, const uint32_t* o, float mul, int lane) {
    constexpr int C = N / 8;                             // pieces of a row, lanes of a group
    static_assert(C == 2 || C == 4, "16 or 32 columns");
    uint4 v[C];
#pragma unroll
    for (int c = 0; c < C; ++c) {
        v[c].x = pack_bf16(__uint_as_float(o[8 * c]) * mul, __uint_as_float(o[8 * c + 1]) * mul);
        v[c].y = pack_bf16(__uint_as_float(o[8 * c + 2]) * mul, __uint_as_float(o[8 * c + 3]) * mul);
        v[c].z = pack_bf16(__uint_as_float(o[8 * c + 4]) * mul, __uint_as_float(o[8 * c + 5]) * mul);
        v[c].w = pack_bf16(__uint_as_float(o[8 * c + 6]) * mul, __uint_as_float(o[8 * c + 7]) * mul);
    }
    // transposition of the group's C x C pieces: lane g ends with piece g of every row of the group
#pragma unroll
    for (int bit = 1; bit < C; bit <<= 1) {
        const bool up = (lane & bit) != 0;
#pragma unroll
        for (int c = 0; c < C; ++c) {
            if (c & bit) continue;
            uint4 &lo = v[c], &hi = v[c | bit];
            const uint4 give = up ? lo : hi;
            uint4 got;
            got.x = __shfl_xor_sync(0xffffffffu, give.x, bit); got.y = __shfl_xor_sync(0xffffffffu, give.y, bit);
            got.z = __shfl_xor_sync(0xffffffffu, give.z, bit); got.w = __shfl_xor_sync(0xffffffffu, give.w, bit);
            if (up) lo = got; else hi = got;
        }
    }
    const int r0 = lane & ~(C - 1);
    __nv_bfloat16* at = row0 + (long long)r0 * stride + (lane & (C - 1)) * 8;
#pragma unroll
    for (int i = 0; i < C; ++i)
        if (r0 + i < rows) *reinterpret_cast<uint4*>(at + i * stride) = v[i];
}

// Host side: tensor map of a [B, H, rows, d] bf16 tensor with element strides (sb, sh, sn, 1) whose box
// is 64 columns x box_rows rows, 128-byte swizzled (one shared-memory panel per box).
bool make_bf16_map(CUtensorMap* map, const void* base, int d, long long rows, int H, int B, long long sn,
                   long long sh, long long sb, int box_rows);
bool tensor_map_encoder_available();
bool make_strip_map(CUtensorMap* map, const void* base, bool is_bf16, int D, long long T, int B, int box_cols, int box_rows);

}  // namespace mka

// Internal declarations shared by the kernels of the FastMKA library (not part of the C ABI).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "mka.h"

namespace mka {

// The kernels of the library are launched so that they may start while the kernel before them in the stream still runs (programmatic
// dependent launch; not the two forms of the session summary that follow a clearing of their scratch): a kernel's CTAs take the SMs' free
// places, set up what needs no memory and wait in chain_wait for the end of the kernel before and for its writes.  One after the other a boundary costs about 2 us of drain, launch and set-up (measured between the
// kernels of a serving step and of a backward), as much as half of the short kernels take.  Nothing in global memory is read or
// written, and no tensor memory allocated (the kernel before may not have taken its own yet), in front of chain_wait;
// chain_trigger stands at the start, since a waiting CTA costs nothing: the next kernel starts when all CTAs of this one have.
// The one exception is the second of the two large backward kernels (tensor cores), which runs beside the first and waits for it at its end
// only.  It may: the first one lets it start only after its own chain_wait and its allocation of tensor memory, so all that the second
// one reads was complete by then (the statistics are read past L1, which may hold an earlier call's); neither reads what the other
// writes, and the forms of a call in which one would (gradients written over keys or values) take the full wait.
__device__ __forceinline__ void chain_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chain_enter() { chain_trigger(); chain_wait(); }

// Launches `kern` in that way; with cluster > 0 as clusters of that many CTAs along x.
template <typename... P, typename... A>
cudaError_t launch_chained(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, int cluster, const A&... args) {
    cudaLaunchAttribute at[2] = {};
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = cluster; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cfg.attrs = at; cfg.numAttrs = cluster > 0 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;
constexpr int kTileM = 128;   // query rows per tile of the tensor-core forward
constexpr int kTileN = 128;   // key rows per tile

// Layout of the caller's workspace: a 256-byte header (device status word first), then the
// per-entry-point scratch.
constexpr size_t kWsHeader = 256;

struct LevelDev {
    const void* k;
    const void* v;
    long long n, sb, sh, sn;
};

struct LevelGradDev {
    void* dk;
    void* dv;
    long long n, sb, sh, sn;
};

struct PagedLevelDev;
struct FwdParams {
    const void* Q;
    void* O;
    float* LSE;         // may be null
    const float* gate;  // [B,T,3]
    LevelDev L[3];
    int B, H, T, d;
    int window, q_offset;
    float scale;        // tau
    int mode;
    int decode;         // every row visible
    int kv_group;       // query heads per KV head (>= 1): head h reads KV head h / kv_group
    int test_stall;     // MKA_FLAG_TEST_STALL (tensor-core forward, dense levels)
    unsigned int* status;   // device status word; the CUDA-core kernel, which waits for nothing, writes MKA_OK itself
    void* scratch;          // room for partial results (tensor-core forward), or null
    size_t scratch_bytes;
    const PagedLevelDev* paged;   // host array of 3, or null: the levels are page pools (tensor-core forward only; L[l].n still holds the rows)
};

template <typename T> struct Elem;
template <> struct Elem<float> {
    static __device__ __forceinline__ float ld(const float* p) { return *p; }
    static __device__ __forceinline__ void st(float* p, float v) { *p = v; }
};
template <> struct Elem<__nv_bfloat16> {
    static __device__ __forceinline__ float ld(const __nv_bfloat16* p) { return __bfloat162float(*p); }
    static __device__ __forceinline__ void st(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }
};

// Rows [lo, hi) of `level` visible to key-timeline position p (L1 causal window, L2 causal prefix,
// L3 everything), clipped to [0, n).
__host__ __device__ __forceinline__ void visible_range(int level, long long p, long long W, long long n,
                                                       int decode, long long& lo, long long& hi) {
    long long a = 0, b = n;
    if (!decode) {
        if (level == 0) { a = p - W + 1; b = p + 1; }
        else if (level == 1) { b = p + 1; }
        if (a < 0) a = 0;
        if (b > n) b = n;
    }
    if (b < a) b = a;
    lo = a; hi = b;
}

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// ---- launchers implemented in the .cu files (all return a cudaError_t from the launch) ----
cudaError_t launch_router(const void* R, const float* W_r, const float* b_r, long long rows, int D, int r_dtype,
                          int route, float* gate, float* log2_gate, int8_t* idx, cudaStream_t st);
cudaError_t launch_fwd_simt(const FwdParams& p, int dtype, cudaStream_t st);

struct DecodeParams {
    const void* q;
    void* O;
    float* LSE;
    const float* gate;   // [B,3]
    LevelDev L[3];
    int B, H, d;
    int kv_group;        // query heads per KV head (>= 1)
    float scale;
    long long chunk_rows;
    long long n_chunks[3];
    long long total_chunks;
    float* partial;      // [B*H, total_chunks, d+2]
    int counted;         // combine: entry 0 of a (batch, head) holds the number of partials that follow, which carry the gate already
    int expected;        // counted: partials of a (batch, head) in a batch of equal lengths
    unsigned int* status;   // device status word that the combine kernel sets to MKA_OK, or null (kernels before it may wait and set it)
};
cudaError_t launch_decode(const DecodeParams& p, cudaStream_t st);
cudaError_t launch_decode_combine(const DecodeParams& p, cudaStream_t st);   // second kernel alone (gate, n_chunks, partial, O, LSE)

struct PagedLevelDev {
    const void* k;
    const void* v;
    const int* table;    // [B, table_stride]
    const int* rows;     // [B] or null
    long long n, table_stride, table_head_stride, sp, sh, sn;
    long long pool_pages; // pages in the pool (needed by the paged forward only)
    int page_shift;      // log2(page_rows)
};
struct DecodePagedParams {
    const void* q;
    const float* gate;   // [B,3]
    PagedLevelDev L[3];
    int B, H, H_kv, d;
    float scale;
    long long chunk_rows;
    long long n_chunks[3];
    long long total_chunks;
    float* partial;      // [B*H, total_chunks, d+2]
    int test_stall;                    // MKA_FLAG_TEST_STALL (copy-engine form): every CTA's producer leaves out the last tile of its share
    int dealt;                         // the copy-engine form: total_chunks = entries per query head (a count, then the partials)
    int few;                           // copy-engine form: few enough sequences and tiles for the short way to a CTA's share
    int deal_shift;                    // copy-engine form: log2 of the sequences in a block of its sums
    unsigned int* status;              // device status word of the call's workspace (bounded waits of the copy-engine form)
    unsigned long long wait_limit_ns;
};
constexpr int kDealCtas = 148 * 2;     // CTAs of the copy-engine form: two per SM
bool decode_paged_dealt(const DecodePagedParams& p);
cudaError_t launch_decode_paged(const DecodePagedParams& p, cudaStream_t st);
cudaError_t launch_l3_index(const void* k, long long n_pages, int H_kv, int page_rows, int d, long long sp, long long sh,
                            long long sn, const float* proj, int bits, unsigned int* codes, cudaStream_t st);
cudaError_t launch_l3_retrieve(const void* q, int B, int H, int H_kv, int d, const float* proj, int bits,
                               const unsigned int* codes, const int* bank, const int* bank_len, long long bank_stride,
                               int max_bank, int R, int page_rows, int* table, int* n_sel, int* rows, cudaStream_t st);

struct BwdParams {
    const void *Q, *O, *dO;
    const float* LSE;
    const float* gate;
    LevelDev L[3];
    LevelGradDev dL[3];
    void* dQ;
    float* dG;        // [B,T,3]
    float* delta;     // ws: [B,H,T]
    float* Gpart;     // ws: [B,H,T,3]
    float* stats;     // ws: room for 6 x [B,H,Tpad] floats (tensor-core path uses 4; Tpad = T rounded up to 128)
    int B, H, T, d;
    int window, q_offset;
    float scale;
    int kv_group;     // query heads per KV head (>= 1); > 1 only on the tensor-core path
    unsigned int* status;   // first 16 bytes of the workspace (status word, tickets): cleared by the first kernel of the call
    int in_place;     // a gradient of keys or values lies in memory of keys or values
    int dg_last;      // dG lies in memory that the call still reads: its sums have to wait for the end of dK and dV
    int test_stall;   // MKA_FLAG_TEST_STALL (tensor-core path): the dK/dV kernel's loader leaves out its last query tile
};
cudaError_t launch_bwd_simt(const BwdParams& p, int dtype, cudaStream_t st);
cudaError_t launch_router_bwd(const void* R, int r_dtype, const float* dG, long long rows, int D, float* dW_r,
                              float* db_r, float* partial, double* db_partial, int n_row_chunks, cudaStream_t st);

cudaError_t launch_fuse_kv(const LevelDev L[3], const LevelGradDev& out, const float* gate, int B, int H, long long n, int d,
                           long long dst_offset, int dtype, cudaStream_t st, const int* dst_table = nullptr,
                           long long dst_table_stride = 0, int dst_page_shift = 0, const int* dst_offsets = nullptr);
cudaError_t launch_l2_summary(const void* X, void* M2, float* state, int use_state, long long n_prev, int B, long long T, int D,
                              int dtype, int kind, float beta, unsigned int* status, cudaStream_t st);
size_t l2_summary_seg_workspace(int B, long long T, int D, int dtype);
cudaError_t launch_l2_summary_seg(const void* X, void* M2, float* state, int use_state, long long n_prev, int B, long long T,
                                  int D, int dtype, int kind, float beta, unsigned int* status, void* scratch, cudaStream_t st);
cudaError_t launch_bwd_dgate(const float* Gpart, int B, int H, long long T, float* dG, cudaStream_t st);
// dG[b,t,l] = sum_h G[b,h,t,l], added up in the order of the heads; at = t * 3 + l.
__device__ __forceinline__ void sum_dgate(const float* Gpart, float* dG, int H, long long T, long long b, long long at) {
    float s = 0.f;
#pragma unroll 8
    for (int h = 0; h < H; ++h) s += __ldcg(Gpart + (b * H + h) * T * 3 + at);
    dG[b * T * 3 + at] = s;
}
// Tensor-core (TMA + tcgen05) backward; same contract as the forward below.
cudaError_t launch_bwd_tc(const BwdParams& p, unsigned int* status_word, cudaStream_t st);
bool bwd_tc_eligible(const BwdParams& p, int dtype);

// Tensor-core (TMA + tcgen05) forward; returns cudaErrorNotSupported when the shape is not eligible.
cudaError_t launch_fwd_tc(const FwdParams& p, unsigned int* status_word, cudaStream_t st);
bool fwd_tc_eligible(const FwdParams& p, int dtype);
size_t fwd_tc_scratch_bytes(const FwdParams& p);      // scratch with which the call would run faster, 0: none

}  // namespace mka

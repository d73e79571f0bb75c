// L3 recall (Alg. 2 step 4, "L3 <- Retrieve(Q_h)"; the method section's vectorized hashing with chunk-based recall).
// The paper names the mechanism but not the hash.  Here a chunk is one page of the long-term key pool and its
// signature is a sign-random-projection code of the SUM of its keys; a query's code comes from the sum of the query
// heads that share the KV head; the R chunks whose codes agree with the query's in the most bits are recalled (ties
// to the earlier chunk) and listed in bank order as a page table for the paged decode.
// Code bits are decided by fp32 arithmetic, so its order is fixed: sums run row by row, a projection is one fmaf
// chain over the columns.
//   l3_index_kernel     HBM-bound: reads every key of the pool once, writes bits/8 bytes per (page, KV head)
//   l3_retrieve_kernel  one CTA per (sequence, KV head): query code, Hamming scores of the bank, a binary search for the R-th best
#include "tc_ptx.cuh"

namespace mka {
namespace {

constexpr int kIdxThreads = 128;                      // threads that project; the two-phase form: all threads
constexpr int kIdxPairs = 64;                         // (page, head) pairs per batch of a CTA: two per lane in the projections
constexpr int kPhasePairs = 32;                       // the same in the two-phase form: one per lane
constexpr int kIdxBitsPerWarp = 16;                   // code bits one warp works out per pass

// 16 bytes that nobody reads again: they leave the L1 to the loads in flight (109 us with plain loads in the form for large pools; the
// other forms, whose pools may still lie in the L2 cache, gain nothing).
__device__ __forceinline__ uint4 ld_once(const void* p) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}

struct L3IndexParams {
    const __nv_bfloat16* k;
    const float* proj;       // [bits, d]
    unsigned int* codes;     // [pages, H_kv, bits / 32]
    long long n_pages, sp, sh, sn;
    int H_kv, page_rows, d, bits;
};

constexpr __host__ __device__ int idx_pitch(int d, bool swaps) { return swaps ? d : d + 4; }

// Dynamic shared memory: projT [d][bits + 4] floats (16 consecutive bits of one column are four broadcast reads), then two
// buffers s [kIdxPairs][idx_pitch] floats (the key sums).  With rows of d + 4 floats the 16-byte reads of eight lanes fall on different
// banks; SWAPS (256 bits, d = 128, sixteen loading warps): four columns of row r lie at place c ^ (r & 7) instead of c.  Padded there too, the SM's shared memory would go
// past 196 KB, and with 228 set aside the L1 cache has half of the room for loads in flight ([7629 pages, 4 heads, 64 rows, 128] 124 -> 158 us).
// Elsewhere the exchange costs more than it gives (1.00 to 1.05 of the time).
// A batch = 64 (page, head) pairs.  The first LOADERS threads load: 16 of them cover one 256-byte row, a thread sums its eight
// columns row by row, with up to 24 (512 loaders: 16) loads in flight across items and batches.  Four more warps project: lane = two pairs,
// warp = 16 bits; four columns cost two 16-byte reads of s, 16 broadcast reads of projT and 128 fmaf.  The two sides work on different batches,
// so the loads of one run under the projections of the other.  As two phases of the same warps, and with one pair to a
// lane, the shared-memory pipe was busy for 78 us and HBM idle half of the time: 147 us (3.6 TB/s) for [32769 pages, 4 heads, 16
// rows, 128] at 64 bits, 123 us with four loading warps in each of two CTAs (registers moved to them from the projecting ones);
// sixteen in one CTA: see many_loaders.
template <int DH, int LOADERS, bool SWAPS = false>
__global__ void __launch_bounds__(LOADERS + kIdxThreads, LOADERS == 128 ? 2 : 1) l3_index_kernel(const L3IndexParams p) {
    chain_enter();
    extern __shared__ __align__(16) float sm[];
    const int ppitch = p.bits + 4;                             // floats between columns of projT (keeps the fill off one bank)
    constexpr int pitch = idx_pitch(DH, SWAPS), kSumFloats = kIdxPairs * pitch;
    constexpr int kSwap = SWAPS ? 7 : 0;                                      // lowest bits of a row's number that exchange its columns
    float* projT = sm;
    float* sums = sm + (size_t)DH * ppitch;
    const bool loads = threadIdx.x < LOADERS;
    const int tid = loads ? threadIdx.x : threadIdx.x - LOADERS, lane = tid & 31, warp = tid >> 5;
    for (int e = threadIdx.x; e < DH * p.bits; e += LOADERS + kIdxThreads) {     // e = j * d + i: coalesced reads of proj
        const int j = e / DH, i = e % DH;
        projT[i * ppitch + j] = p.proj[e];
    }
    __syncthreads();
    constexpr int vecs = DH / 8;                               // 16-byte pieces of a row: 16 (d = 128) or 8 (d = 64)
    constexpr int kPerThread = kIdxPairs * vecs / LOADERS; // (pair, piece) items of a thread in a batch: 8 or 4 (512 loaders: 2 or 1)
    constexpr int kSlotStep = LOADERS / vecs;              // pairs between a thread's items
    const long long pairs = p.n_pages * p.H_kv;
    const int words = p.bits / 32;
    const long long step = (long long)gridDim.x * kIdxPairs, first = (long long)blockIdx.x * kIdxPairs;
    // barriers 1, 2: buffer 0 / 1 is filled;  3, 4: it is free again (one side arrives, the other waits)
    auto arrive = [](int id) { asm volatile("bar.arrive %0, %1;" ::"r"(id), "n"(LOADERS + kIdxThreads) : "memory"); };
    auto wait = [](int id) { asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(LOADERS + kIdxThreads) : "memory"); };
    if (loads) {
        if constexpr (LOADERS == 128) asm volatile("setmaxnreg.inc.sync.aligned.u32 152;");  // 256 threads x 128 registers at launch = 128 x 152 + 128 x 104
        const int slot0 = tid / vecs, piece = tid % vecs;
        constexpr int kDepth = LOADERS == 128 ? 3 : 2;
        uint4 u[kDepth][8];
        // the next eight rows to ask for
        long long f_base = first;
        int f_item = 0, f_row = 0;
        const __nv_bfloat16* f_src = nullptr;                  // null: the pair does not exist
        auto locate = [&] {
            const long long pair = f_base + slot0 + f_item * kSlotStep;
            f_src = nullptr;
            if (pair < pairs) {
                const long long page = pair <= 0x7fffffffLL ? (long long)((unsigned)pair / (unsigned)p.H_kv) : pair / p.H_kv;
                f_src = p.k + page * p.sp + (pair - page * p.H_kv) * p.sh + piece * 8;
            }
        };
        locate();
        auto load = [](const __nv_bfloat16* src) {
            if constexpr (LOADERS == 512) return ld_once(src);
            else return __ldg(reinterpret_cast<const uint4*>(src));
        };
        auto fetch = [&](uint4 (&to)[8]) {
            if (f_base >= pairs) return;
            if (f_src) {
                if (f_row + 8 <= p.page_rows) {
#pragma unroll
                    for (int r = 0; r < 8; ++r) to[r] = load(f_src + r * p.sn);
                } else {
#pragma unroll
                    for (int r = 0; r < 8; ++r)
                        if (f_row + r < p.page_rows) to[r] = load(f_src + r * p.sn);
                }
                f_src += 8 * p.sn;
            }
            f_row += 8;
            if (f_row >= p.page_rows) {
                f_row = 0;
                if (++f_item == kPerThread) { f_item = 0; f_base += step; }
                locate();
            }
        };
#pragma unroll
        for (int i = 0; i < kDepth; ++i) fetch(u[i]);
        unsigned long long acc[4];                             // eight columns as packed pairs (add.rn.f32x2: two plain sums)
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[i] = 0ull;
        auto add_row = [&](const uint4& v) {
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                unsigned long long x2;
                asm("mov.b64 %0, {%1, %2};" : "=l"(x2) : "r"(w[i] << 16), "r"(w[i] & 0xffff0000u));
                asm("add.rn.f32x2 %0, %0, %1;" : "+l"(acc[i]) : "l"(x2));
            }
        };
        long long base = first;
        int n = 0, item = 0, row = 0;
        while (base < pairs) {
#pragma unroll
            for (int x = 0; x < kDepth; ++x) {
                if (base >= pairs) break;
                if (row + 8 <= p.page_rows) {
#pragma unroll
                    for (int r = 0; r < 8; ++r) add_row(u[x][r]);
                } else {
#pragma unroll
                    for (int r = 0; r < 8; ++r)
                        if (row + r < p.page_rows) add_row(u[x][r]);   // rows past the page add nothing, not even +0
                }
                fetch(u[x]);
                row += 8;
                if (row >= p.page_rows) {
                    if (item == 0 && n >= 2) wait(3 + (n & 1));            // the batch before last has been projected
                    const int slot = slot0 + item * kSlotStep, swap = (slot & kSwap) * 4;
                    float* s = sums + (n & 1) * kSumFloats + slot * pitch;
                    *reinterpret_cast<ulonglong2*>(s + ((piece * 8) ^ swap)) = make_ulonglong2(acc[0], acc[1]);
                    *reinterpret_cast<ulonglong2*>(s + ((piece * 8 + 4) ^ swap)) = make_ulonglong2(acc[2], acc[3]);
#pragma unroll
                    for (int i = 0; i < 4; ++i) acc[i] = 0ull;
                    row = 0;
                    if (++item == kPerThread) {
                        arrive(1 + (n & 1));
                        item = 0; ++n; base += step;
                    }
                }
            }
        }
    } else {
        if constexpr (LOADERS == 128) asm volatile("setmaxnreg.dec.sync.aligned.u32 104;");
        unsigned short* codes16 = reinterpret_cast<unsigned short*>(p.codes);
        int n = 0;
        for (long long base = first; base < pairs; base += step, ++n) {
            // ---- projections: one fmaf chain per (pair, bit) over the columns 0..d-1
            wait(1 + (n & 1));
            const float* sv = sums + (n & 1) * kSumFloats + lane * pitch;
            const int swap = (lane & kSwap) * 4;                               // (of row lane + 32 too)
            for (int j0 = warp * kIdxBitsPerWarp; j0 < p.bits; j0 += (kIdxThreads / 32) * kIdxBitsPerWarp) {
                // two chains per instruction (fma.rn.f32x2: each half is the same correctly rounded fma as fmaf)
                unsigned long long a2[2][kIdxBitsPerWarp / 2];
#pragma unroll
                for (int q = 0; q < 2; ++q)
#pragma unroll
                    for (int j = 0; j < kIdxBitsPerWarp / 2; ++j) a2[q][j] = 0ull;          // two +0.f
                const float* pj = projT + j0;
                // 32 columns to a turn: a warp has its scheduler's share to itself and waits for the reads at the start of each turn (the loading warps never
                // wait for long: they ran out of buffers for 2 % of the time, these warps of sums for 0.1 %).  Turns of 4 / 8 / 16 / 32 columns:
                // [32769 pages, 4 heads, 16 rows, 128], 64 bits 118 / 111 / 111 / 109.5 us; 128 bits [20000, 8, 16, 128] 204 / 190 / 183 / 182;
                // 256 bits [20000, 2, 8, 128] 93.0 / 89.3 / 85.4 / 81.9.
#pragma unroll 8
                for (int i4 = 0; i4 < DH; i4 += 4) {
                    const float4 xa4 = *reinterpret_cast<const float4*>(sv + (i4 ^ swap)), xb4 = *reinterpret_cast<const float4*>(sv + 32 * pitch + (i4 ^ swap));
                    const float xa[4] = {xa4.x, xa4.y, xa4.z, xa4.w}, xb[4] = {xb4.x, xb4.y, xb4.z, xb4.w};
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        unsigned long long x2[2];
                        asm("mov.b64 %0, {%1, %1};" : "=l"(x2[0]) : "f"(xa[k]));
                        asm("mov.b64 %0, {%1, %1};" : "=l"(x2[1]) : "f"(xb[k]));
#pragma unroll
                        for (int v = 0; v < kIdxBitsPerWarp / 4; ++v) {
                            const ulonglong2 pr = *reinterpret_cast<const ulonglong2*>(pj + (size_t)(i4 + k) * ppitch + 4 * v);   // bits 4v..4v+3 of the column
#pragma unroll
                            for (int q = 0; q < 2; ++q) {
                                asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(a2[q][2 * v]) : "l"(pr.x), "l"(x2[q]));
                                asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(a2[q][2 * v + 1]) : "l"(pr.y), "l"(x2[q]));
                            }
                        }
                    }
                }
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    unsigned half = 0u;
#pragma unroll
                    for (int j = 0; j < kIdxBitsPerWarp / 2; ++j) {
                        float lo, hi;
                        asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a2[q][j]));
                        half |= (lo >= 0.f ? 1u : 0u) << (2 * j);
                        half |= (hi >= 0.f ? 1u : 0u) << (2 * j + 1);
                    }
                    // bits j0..j0+15 are one 16-bit half of word j0 / 32 (low half first)
                    const long long pair = base + q * 32 + lane;
                    if (pair < pairs) codes16[(pair * words) * 2 + j0 / 16] = (unsigned short)half;
                }
            }
            if (base + 2 * step < pairs) arrive(3 + (n & 1));  // (nobody waits for the last two)
        }
    }
}

// The same in two phases: all 128 threads load and sum a batch of 32 pairs, then all project it, lane = pair.  No thread is set aside for
// projections and up to four CTAs share an SM, so this form is for pools with few code bits to a key row and for small ones
// (see launch_l3_index).
// Dynamic shared memory: projT [d][bits + 4] floats, then s [kPhasePairs][d + 1] floats.
template <int DH>
__global__ void __launch_bounds__(kIdxThreads, 4) l3_index_phases_kernel(const L3IndexParams p) {
    chain_enter();
    extern __shared__ __align__(16) float sm[];
    const int ppitch = p.bits + 4;                             // floats between columns of projT (keeps the fill off one bank)
    float* projT = sm;
    float* s = sm + (size_t)DH * ppitch;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int pitch = DH + 1;
    for (int e = tid; e < DH * p.bits; e += kIdxThreads) {     // e = j * d + i: coalesced reads of proj
        const int j = e / DH, i = e % DH;
        projT[i * ppitch + j] = p.proj[e];
    }
    constexpr int vecs = DH / 8;                               // 16-byte pieces of a row: 16 (d = 128) or 8 (d = 64)
    constexpr int items = kPhasePairs * vecs;                    // (pair, piece) items of a batch
    constexpr int kPerThread = items / kIdxThreads;            // 4 or 2: taken two at a time, 16 loads in flight
    const long long pairs = p.n_pages * p.H_kv;
    const int words = p.bits / 32;
    unsigned short* codes16 = reinterpret_cast<unsigned short*>(p.codes);
    for (long long base = (long long)blockIdx.x * kPhasePairs; base < pairs; base += (long long)gridDim.x * kPhasePairs) {
        __syncthreads();                                       // projT is there; the previous batch is done with s
        // ---- sums of the pages' keys, row by row
#pragma unroll
        for (int k0 = 0; k0 < kPerThread; k0 += 2) {
            float acc[2][8];
            const __nv_bfloat16* src[2];
            bool live[2];
            int slot[2], piece[2];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int it = tid + (k0 + q) * kIdxThreads;
                slot[q] = it / vecs; piece[q] = it % vecs;
                const long long pair = base + slot[q];
                live[q] = pair < pairs;
                const long long pc = live[q] ? pair : 0;
                src[q] = p.k + (pc / p.H_kv) * p.sp + (pc % p.H_kv) * p.sh + piece[q] * 8;
#pragma unroll
                for (int i = 0; i < 8; ++i) acc[q][i] = 0.f;
            }
            for (int r0 = 0; r0 < p.page_rows; r0 += 8) {
                uint4 u[2][8];
#pragma unroll
                for (int q = 0; q < 2; ++q)
#pragma unroll
                    for (int r = 0; r < 8; ++r)
                        u[q][r] = (live[q] && r0 + r < p.page_rows)
                                      ? __ldg(reinterpret_cast<const uint4*>(src[q] + (long long)(r0 + r) * p.sn))
                                      : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
                for (int q = 0; q < 2; ++q)
#pragma unroll
                    for (int r = 0; r < 8; ++r) {
                        if (r0 + r < p.page_rows) {                // rows past the page add nothing, not even +0
                            const uint32_t w[4] = {u[q][r].x, u[q][r].y, u[q][r].z, u[q][r].w};
#pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                acc[q][2 * i] = acc[q][2 * i] + __uint_as_float(w[i] << 16);
                                acc[q][2 * i + 1] = acc[q][2 * i + 1] + __uint_as_float(w[i] & 0xffff0000u);
                            }
                        }
                    }
            }
#pragma unroll
            for (int q = 0; q < 2; ++q)
#pragma unroll
                for (int i = 0; i < 8; ++i) s[slot[q] * pitch + piece[q] * 8 + i] = acc[q][i];
        }
        __syncthreads();
        // ---- projections: one fmaf chain per (pair, bit) over the columns 0..d-1
        const long long pair = base + lane;
        const float* sv = s + lane * pitch;
        for (int j0 = warp * kIdxBitsPerWarp; j0 < p.bits; j0 += (kIdxThreads / 32) * kIdxBitsPerWarp) {
            // two chains per instruction (fma.rn.f32x2: each half is the same correctly rounded fma as fmaf)
            unsigned long long a2[kIdxBitsPerWarp / 2];
#pragma unroll
            for (int j = 0; j < kIdxBitsPerWarp / 2; ++j) a2[j] = 0ull;          // two +0.f
            const float* pj = projT + j0;
            for (int i = 0; i < DH; ++i) {
                const float x = sv[i];
                unsigned long long x2;
                asm("mov.b64 %0, {%1, %1};" : "=l"(x2) : "f"(x));
#pragma unroll
                for (int v = 0; v < kIdxBitsPerWarp / 4; ++v) {
                    const ulonglong2 pr = *reinterpret_cast<const ulonglong2*>(pj + (size_t)i * ppitch + 4 * v);   // bits 4v..4v+3 of column i
                    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(a2[2 * v]) : "l"(pr.x), "l"(x2));
                    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(a2[2 * v + 1]) : "l"(pr.y), "l"(x2));
                }
            }
            unsigned half = 0u;
#pragma unroll
            for (int j = 0; j < kIdxBitsPerWarp / 2; ++j) {
                float lo, hi;
                asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a2[j]));
                half |= (lo >= 0.f ? 1u : 0u) << (2 * j);
                half |= (hi >= 0.f ? 1u : 0u) << (2 * j + 1);
            }
            // bits j0..j0+15 are one 16-bit half of word j0 / 32 (low half first)
            if (pair < pairs) codes16[(pair * words) * 2 + j0 / 16] = (unsigned short)half;
        }
    }
}

struct L3RetrieveParams {
    const __nv_bfloat16* q;       // [B, H, d]
    const float* proj;            // [bits, d]
    const unsigned int* codes;    // [pages, H_kv, words]
    const int* bank;              // [B, bank_stride]
    const int* bank_len;          // [B]
    int* table;                   // [B, H_kv, R]
    int* n_sel;                   // [B] or null
    int* rows;                    // [B] or null: n_sel * page_rows
    long long bank_stride;
    int B, H, H_kv, d, bits, R, page_rows, max_bank;
    int per_cta;                  // chunks that a CTA of the cluster takes at most
    int stage_proj;               // the projection is staged in shared memory (it fits beside the scores and is 16-byte aligned)
    int code_vec;                 // code words fetched by one load: 4 (16-byte aligned codes of 128 or 256 bits), 2 (64 bits, 8-byte aligned) or 1
};

constexpr int kRetThreads = 1024;
constexpr int kRetWarps = kRetThreads / 32;

constexpr int kRetMaxCluster = 8;

// A cluster of CTAs per (sequence, KV head), each with a stretch of the bank.  Everything here is latency: the code words are asked for
// before the query's code is worked out; the R best are not picked one after the other but cut off at once.  A CTA counts its
// chunks by score, the counts of the cluster meet in distributed shared memory, and the R-th best score, what lies above it and
// how much of both the CTAs in front hold come from one scan over them; inside a CTA per-group counts and their scan give every
// recalled chunk its place in bank order.  The gather of the codes is one sector a chunk, which a single SM's L1 works off one a
// cycle: with one CTA and a binary search over the scores (a pass and a barrier each step), 8 of 8192 chunks took 15 us.
// Dynamic shared memory: unsigned short score[per_cta], int before[per_cta / 32 rounded up to whole rounds], the projection.
__global__ void __launch_bounds__(kRetThreads) l3_retrieve_kernel(const L3RetrieveParams p) {
    extern __shared__ __align__(16) unsigned short score[];
    __shared__ __align__(16) float qs[256];
    __shared__ __align__(16) unsigned int qcode[8];
    __shared__ int hist[257], total[257], lower[257];          // chunks by score: this CTA's, the cluster's, those of the CTAs in front
    __shared__ int cut_s[4];
    chain_enter();
    int rank, size;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(size));
    int* before = reinterpret_cast<int*>(score + (p.per_cta + 7) / 8 * 8);
    float* projs = reinterpret_cast<float*>(before + (p.per_cta + kRetThreads - 1) / kRetThreads * kRetWarps);   // [bits][d + 4]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int list = blockIdx.x / size, b = list / p.H_kv, kvh = list % p.H_kv;
    const int G = p.H / p.H_kv, words = p.bits / 32;
    int n_bank = p.bank_len[b];
    n_bank = n_bank < 0 ? 0 : (n_bank > p.max_bank ? p.max_bank : n_bank);
    const int per = ((n_bank + size - 1) / size + 31) / 32 * 32;            // at most per_cta
    const int c_first = min(rank * per, n_bank), n = min(per, n_bank - c_first);   // this CTA's chunks, from here on counted from its first
    const int* bank = p.bank + (long long)b * p.bank_stride + c_first;
    for (int i = tid; i <= p.bits; i += kRetThreads) hist[i] = 0;
    // 64-bit codes: the first eight chunks of a thread, page numbers first, then all code words.  (Wider codes would need 32 and
    // 64 registers for that, half or all of what a thread has here; theirs are asked for after the query's code.)
    constexpr int kAhead = 8;
    uint2 ahead[kAhead];
    if (p.code_vec == 2) {
        int page[kAhead];
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
            const int c = tid + u * kRetThreads;
            page[u] = c < n ? bank[c] : -1;
        }
#pragma unroll
        for (int u = 0; u < kAhead; ++u)
            ahead[u] = page[u] >= 0 ? __ldg(reinterpret_cast<const uint2*>(p.codes + ((long long)page[u] * p.H_kv + kvh) * 2)) : make_uint2(0u, 0u);
    }
    // the projection, where there is room for it: its rows are read by one thread each, four columns at a time
    const int pitch = p.d + 4;
    if (p.stage_proj)
        for (int e = tid * 4; e < p.bits * p.d; e += kRetThreads * 4)
            *reinterpret_cast<float4*>(projs + (e / p.d) * pitch + e % p.d) = __ldg(reinterpret_cast<const float4*>(p.proj + e));
    // query of the KV head: the group's heads summed in head order, fp32
    if (tid < p.d) {
        const __nv_bfloat16* q0 = p.q + ((long long)b * p.H + (long long)kvh * G) * p.d + tid;
        float acc = 0.f;
        for (int g0 = 0; g0 < G; g0 += 8) {
            float x[8];
#pragma unroll
            for (int g = 0; g < 8; ++g) x[g] = g0 + g < G ? __bfloat162float(q0[(long long)(g0 + g) * p.d]) : 0.f;
#pragma unroll
            for (int g = 0; g < 8; ++g)
                if (g0 + g < G) acc = acc + x[g];
        }
        qs[tid] = acc;
    }
    __syncthreads();
    if (tid < p.bits) {                                        // whole warps: bits is a multiple of 32
        const float* pr = p.proj + (long long)tid * p.d;
        float acc = 0.f;
        if (p.stage_proj) {
#pragma unroll 8
            for (int i = 0; i < p.d; i += 4) {
                const float4 v = *reinterpret_cast<const float4*>(projs + tid * pitch + i), x = *reinterpret_cast<const float4*>(qs + i);
                acc = fmaf(v.x, x.x, acc); acc = fmaf(v.y, x.y, acc); acc = fmaf(v.z, x.z, acc); acc = fmaf(v.w, x.w, acc);
            }
        } else {
            for (int i = 0; i < p.d; ++i) acc = fmaf(pr[i], qs[i], acc);
        }
        const unsigned int word = __ballot_sync(0xffffffffu, acc >= 0.f);
        if (lane == 0) qcode[warp] = word;
    }
    __syncthreads();
    // agreement of every chunk's code with the query's: 0..bits (<= 256)
    if (p.code_vec == 2) {
        const unsigned int q0 = qcode[0], q1 = qcode[1];
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
            const int c = tid + u * kRetThreads;
            if (c >= n) continue;
            const int sc = p.bits - __popc(ahead[u].x ^ q0) - __popc(ahead[u].y ^ q1);
            score[c] = (unsigned short)sc;
            atomicAdd(&hist[sc], 1);
        }
    }
    // All words of a code lie in one sector, so they are fetched together: word by word over eight chunks, a CTA's 8192 sectors had
    // left its L1 before the next word (whole kernel, 256 bits, 40,000 chunks: 366 us; one after the other and 32 bits a load 221; now 110).
    const unsigned int* codes = p.codes + (long long)kvh * words;
    const long long page_words = (long long)p.H_kv * words;
    for (int c0 = tid + (p.code_vec == 2 ? kAhead * kRetThreads : 0); c0 < n; c0 += 8 * kRetThreads) {
        int page[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int c = c0 + u * kRetThreads;
            page[u] = c < n ? bank[c] : 0;
        }
        auto put = [&](int u, int dist) {
            const int c = c0 + u * kRetThreads;
            if (c >= n) return;
            score[c] = (unsigned short)(p.bits - dist);
            atomicAdd(&hist[p.bits - dist], 1);
        };
        if (p.code_vec == 4) {
            const uint4 qa = *reinterpret_cast<const uint4*>(qcode), qb = *reinterpret_cast<const uint4*>(qcode + 4);
            auto differ = [](const uint4& x, const uint4& y) { return __popc(x.x ^ y.x) + __popc(x.y ^ y.y) + __popc(x.z ^ y.z) + __popc(x.w ^ y.w); };
#pragma unroll
            for (int u0 = 0; u0 < 8; u0 += 4) {
                uint4 a[4], b[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const uint4* at = reinterpret_cast<const uint4*>(codes + page[u0 + u] * page_words);
                    a[u] = __ldg(at);
                    b[u] = words == 8 ? __ldg(at + 1) : qb;
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) put(u0 + u, differ(a[u], qa) + differ(b[u], qb));
            }
        } else if (p.code_vec == 2) {
            uint2 w[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) w[u] = __ldg(reinterpret_cast<const uint2*>(codes + page[u] * page_words));
#pragma unroll
            for (int u = 0; u < 8; ++u) put(u, __popc(w[u].x ^ qcode[0]) + __popc(w[u].y ^ qcode[1]));
        } else {
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                int dist = 0;
                for (int w = 0; w < words; ++w) dist += __popc(__ldg(codes + page[u] * page_words + w) ^ qcode[w]);
                put(u, dist);
            }
        }
    }
    // (a thread reads back only the scores it wrote, up to the barriers below)
    const int k = p.R < n_bank ? p.R : n_bank;
    const int rounds = (n + kRetThreads - 1) / kRetThreads;
    __syncthreads();
    cluster_sync();                                            // every CTA's counts are there
    for (int i = tid; i <= p.bits; i += kRetThreads) {
        int sum = 0, front = 0;
        int v[kRetMaxCluster];                                 // all reads at once, a missing CTA's from the first one
#pragma unroll
        for (int r = 0; r < kRetMaxCluster; ++r) v[r] = __float_as_int(ld_cluster(smem_u32(&hist[i]), r < size ? r : 0));
#pragma unroll
        for (int r = 0; r < kRetMaxCluster; ++r) {
            sum += r < size ? v[r] : 0;
            front += r < rank ? v[r] : 0;
        }
        total[i] = sum; lower[i] = front;
    }
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");           // (waited for at the end: nobody leaves while its counts are read)
    __syncthreads();
    // the largest score that at least k chunks reach, how many are above it, and how many above and at it the CTAs in front hold
    if (warp == 0) {
        int above = 0, above_front = 0;
        for (int top = p.bits; top >= 0; top -= 32) {          // lane = score top - lane
            const int at = top - lane, own = at >= 0 ? total[at] : 0, own_front = at >= 0 ? lower[at] : 0;
            int sum = own, front = own_front;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int x = __shfl_up_sync(0xffffffffu, sum, o), y = __shfl_up_sync(0xffffffffu, front, o);
                if (lane >= o) { sum += x; front += y; }
            }
            const unsigned int reach = __ballot_sync(0xffffffffu, above + sum >= k);
            if (reach) {
                if (lane == __ffs(reach) - 1) {
                    cut_s[0] = at; cut_s[1] = above + sum - own;
                    cut_s[2] = above_front + front - own_front; cut_s[3] = own_front;
                }
                break;
            }
            above += __shfl_sync(0xffffffffu, sum, 31);
            above_front += __shfl_sync(0xffffffffu, front, 31);
        }
    }
    __syncthreads();
    const int lo = cut_s[0], at_cut = k - cut_s[1];            // the cut, and how many of the chunks at it are recalled
    // per group of 32 chunks, in bank order: chunks above the cut (low half) and at it (high half)
    for (int r = 0; r < rounds; ++r) {
        const int c = r * kRetThreads + tid;
        const int sc = c < n ? score[c] : -1;
        const unsigned int gt = __ballot_sync(0xffffffffu, sc > lo), eq = __ballot_sync(0xffffffffu, sc == lo);
        if (lane == 0) before[r * kRetWarps + warp] = __popc(gt) | (__popc(eq) << 16);
    }
    __syncthreads();
    // what comes before each group (fewer than 64 above the cut; at it: saturated at k): a warp scans the groups of one round,
    // then every warp adds up the rounds before its own
    __shared__ int total_gt[96], total_eq[96];                 // (at most 96 rounds: 98304 chunks)
    for (int r = warp; r < rounds; r += kRetWarps) {
        const int v = before[r * kRetWarps + lane];
        int gt = v & 0xffff, eq = v >> 16;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int g = __shfl_up_sync(0xffffffffu, gt, o), e = __shfl_up_sync(0xffffffffu, eq, o);
            if (lane >= o) { gt += g; eq += e; }
        }
        if (lane == 31) { total_gt[r] = gt; total_eq[r] = eq; }
        const int eq_before = eq - (v >> 16);
        before[r * kRetWarps + lane] = (gt - (v & 0xffff)) | ((eq_before < k ? eq_before : k) << 16);
    }
    __syncthreads();
    int* out = p.table + ((long long)b * p.H_kv + kvh) * p.R;
    int run_gt = cut_s[2], run_eq = min(cut_s[3], at_cut);     // (past at_cut the exact number does not matter)
    for (int r = 0; r < rounds; ++r) {
        const int c = r * kRetThreads + tid;
        const int sc = c < n ? score[c] : -1;
        const unsigned int gt = __ballot_sync(0xffffffffu, sc > lo), eq = __ballot_sync(0xffffffffu, sc == lo);
        const int round_gt = run_gt, round_eq = run_eq;
        run_gt += total_gt[r];
        run_eq += total_eq[r];
        if (sc < lo) continue;
        const unsigned int below = (1u << lane) - 1u;
        const int v = before[r * kRetWarps + warp];
        const int gt_before = round_gt + (v & 0xffff) + __popc(gt & below), eq_before = round_eq + (v >> 16) + __popc(eq & below);
        if (sc > lo || eq_before < at_cut) out[gt_before + (eq_before < at_cut ? eq_before : at_cut)] = bank[c];   // bank (time) order
    }
    if (rank == 0)
        for (int i = k + tid; i < p.R; i += kRetThreads) out[i] = 0;
    if (tid == 0 && kvh == 0 && rank == 0) {
        if (p.n_sel) p.n_sel[b] = k;
        if (p.rows) p.rows[b] = k * p.page_rows;
    }
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

// Sixteen loading warps in a CTA that has its SM to itself, instead of eight in two CTAs: half of the warp cycles of the eight went
// into the adds' latencies with their loads not yet asked for again (DRAM 53 % busy), and the two CTAs' copies of the projection take
// the room of loads in flight.  The four projecting warps then serve twice the rows, so the form is for few code bits to a row, and for pools
// that give its CTAs a batch of 64 pairs.  Time of the better of the two other forms over its, 4 KV heads, pages of 16 / 24 / 32 / 64 rows, 300 MB of keys:
//   d = 64    32 bits 1.09 / 1.12 / 1.05 / 0.99    64 bits 1.16 / 1.23 / 1.11 / 1.05    128 bits 0.93 / 1.16 / 1.25 / 1.18    256 bits 0.91 / 1.01 / 0.99 / 1.27
//   d = 128           1.15 / 1.10 / 1.07 / 0.99            1.25 / 1.37 / 1.33 / 1.30             1.31 / 1.65 / 1.63 / 1.36             0.96 / 1.12 / 1.34 / 1.74
// and over those pages by size, in the L2 cache and not: 64 and 128 bits, 20 to 60 MB 0.99 .. 2.09, 90 and 150 MB 0.96 .. 2.2, 5 MB 0.83 .. 1.5; 256 bits,
// 40 to 150 MB 0.95 .. 1.8, 20 MB 0.93 .. 1.7; 32 bits, 20 to 60 MB 0.84 .. 1.5, 90 and 150 MB 0.84 .. 1.13 (d = 64), 1.00 .. 1.5 (d = 128).
// Pages of 8 rows from 90 MB on 0.86 .. 1.14.  Over 560 sizes of 5 to 500 MB, no pick is slower than with the line at 80 MB, where it lay before the projecting
// warps took longer turns, and those between the lines are up to twice as fast ([1831 pages, 4 heads, 32 rows, 128], 64 bits: 23.8 -> 12.5 us).
// [32769 pages, 4 heads, 16 rows, 128], 64 bits: 117 us with eight loading warps, 104 with sixteen.
bool many_loaders(const L3IndexParams& p) {
    if (p.page_rows < 16 || p.bits > (p.d == 128 ? 11 : (p.page_rows >= 24 ? 8 : 4)) * p.page_rows) return false;
    const double from = p.bits == 32 ? (p.d == 128 ? 80e6 : 200e6) : (p.d == 64 && p.page_rows < 24 ? 80e6 : (p.bits == 256 ? 30e6 : 15e6));
    return (double)p.n_pages * p.H_kv * p.page_rows * p.d * 2.0 >= from;
}

// Which of the two others.  The one with projecting warps of its own wins where projections are a good part of the work and
// there are batches enough for all SMs; where a key row carries few code bits (its projecting half idles; at 32 bits two of those four
// warps never have work, at 128 bits and d = 128 one CTA fits an SM) and for small pools the two-phase form does.  Time of the
// first over that of the second, 20 to 500 MB of keys, 4 KV heads (the lines matter below and beside those of many_loaders only):
//   d = 64    32 bits, pages of 8 to 64 rows     1.04 .. 1.7            d = 128   32 bits    1.03 .. 1.6
//             64 bits, 8 / 16 rows               0.74 .. 0.97                     64 bits, 8 / 16 rows     0.68 .. 0.96
//             64 bits, 24 / 32 / 64 rows         0.93 .. 1.12 / 1.02 .. 1.23 / 1.15 .. 1.49                0.88 .. 0.92 / 0.93 .. 1.02 / 0.99 .. 1.21
//             128 bits, 24 / 32 / 64 rows        0.82 .. 0.89 / 0.90 .. 0.99 / 1.03 .. 1.26                0.84 .. 1.04 / 0.97 .. 1.18 / 1.39 .. 1.54
//             256 bits, 16 / 64 rows             0.45 .. 0.84 / 0.65 .. 1.08                               0.52 .. 0.85 / 0.88 .. 0.96
//   pools of at most 74 batches of 64 pairs      0.97 .. 1.87                                              0.89 .. 1.58
bool two_phases(const L3IndexParams& p) {
    if (p.bits == 32 || p.n_pages * p.H_kv <= 74 * kIdxPairs) return true;
    return (p.bits == 64 && p.page_rows >= 24) || (p.bits == 128 && p.page_rows >= 32);
}

}  // namespace

cudaError_t launch_l3_index(const void* k, long long n_pages, int H_kv, int page_rows, int d, long long sp, long long sh,
                            long long sn, const float* proj, int bits, unsigned int* codes, cudaStream_t st) {
    if (n_pages == 0 || H_kv == 0) return cudaSuccess;
    L3IndexParams p;
    p.k = static_cast<const __nv_bfloat16*>(k); p.proj = proj; p.codes = codes;
    p.n_pages = n_pages; p.sp = sp; p.sh = sh; p.sn = sn; p.H_kv = H_kv; p.page_rows = page_rows; p.d = d; p.bits = bits;
    // persistent CTAs: every CTA transposes the projection into shared memory once and then walks its batches
    // (the grid is shrunk so that all CTAs get the same number of batches)
    auto launch = [&](auto kern, int batch, int buffers, int pitch, int threads, auto ctas_per_sm) {
        const size_t smem = ((size_t)d * (bits + 4) + (size_t)buffers * batch * pitch) * sizeof(float);
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        const long long batches = (n_pages * H_kv + batch - 1) / batch, resident = 148LL * ctas_per_sm(smem);
        const long long per_cta = (batches + resident - 1) / resident, grid = (batches + per_cta - 1) / per_cta;
        return launch_chained(kern, dim3((unsigned)grid), dim3(threads), smem, st, 0, p);
    };
    if (many_loaders(p)) {
        const bool swaps = d == 128 && bits == 256;
        return launch(swaps ? l3_index_kernel<128, 512, true> : (d == 128 ? l3_index_kernel<128, 512> : l3_index_kernel<64, 512>), kIdxPairs, 2,
                      idx_pitch(d, swaps), 512 + kIdxThreads, [](size_t) { return 1; });
    }
    if (two_phases(p))
        return launch(d == 128 ? l3_index_phases_kernel<128> : l3_index_phases_kernel<64>, kPhasePairs, 1, d + 1, kIdxThreads,
                      [](size_t smem) { return smem > 110 * 1024 ? 1 : (smem > 72 * 1024 ? 2 : (smem > 54 * 1024 ? 3 : 4)); });
    return launch(d == 128 ? l3_index_kernel<128, 128> : l3_index_kernel<64, 128>, kIdxPairs, 2, idx_pitch(d, false), 2 * kIdxThreads,
                  [](size_t smem) { return smem > 112 * 1024 ? 1 : 2; });
}

cudaError_t launch_l3_retrieve(const void* q, int B, int H, int H_kv, int d, const float* proj, int bits,
                               const unsigned int* codes, const int* bank, const int* bank_len, long long bank_stride,
                               int max_bank, int R, int page_rows, int* table, int* n_sel, int* rows, cudaStream_t st) {
    if (B == 0 || H_kv == 0) return cudaSuccess;
    L3RetrieveParams p;
    p.q = static_cast<const __nv_bfloat16*>(q); p.proj = proj; p.codes = codes; p.bank = bank; p.bank_len = bank_len;
    p.table = table; p.n_sel = n_sel; p.rows = rows; p.bank_stride = bank_stride;
    p.B = B; p.H = H; p.H_kv = H_kv; p.d = d; p.bits = bits; p.R = R; p.page_rows = page_rows; p.max_bank = max_bank;
    // CTAs of a cluster: a bank of a few thousand chunks is spread until a CTA has about a thousand, while all CTAs fit the chip at once
    int size = 1;
    while (size < kRetMaxCluster && size * 1024 < max_bank && (long long)B * H_kv * size * 2 <= 148) size *= 2;
    p.per_cta = ((max_bank + size - 1) / size + 31) / 32 * 32;
    size_t smem = ((size_t)p.per_cta + 7) / 8 * 8 * sizeof(unsigned short) +
                  ((size_t)p.per_cta + kRetThreads - 1) / kRetThreads * kRetWarps * sizeof(int) + 16;
    const size_t with_proj = smem + (size_t)bits * (d + 4) * sizeof(float);
    const uintptr_t at = reinterpret_cast<uintptr_t>(codes);
    p.code_vec = bits >= 128 && at % 16 == 0 ? 4 : (bits == 64 && at % 8 == 0 ? 2 : 1);
    p.stage_proj = with_proj <= 220 * 1024 && (reinterpret_cast<uintptr_t>(proj) & 15) == 0;
    if (p.stage_proj) smem = with_proj;
    cudaError_t e = cudaFuncSetAttribute(l3_retrieve_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return launch_chained(l3_retrieve_kernel, dim3((unsigned)(B * H_kv * size)), dim3(kRetThreads), smem, st, size, p);
}

}  // namespace mka

// tc_gemm.cuh -- BF16 GEMM on the fifth-generation tensor cores (tcgen05) of sm_103a.
//
//   C[m][n] = act( sum_k A[m][k] * B[n][k] + bias[n] )        ("TN": both operands K-contiguous)
//
// Persistent: one CTA per SM takes 128 x BN output tiles in turn (columns fastest: the CTAs at work
// share A panels and write neighbouring pieces of the same rows; 0.73 against 0.82 ms for the
// product below with rows fastest).  Warp 0 streams 128 x 64 (A) and BN x 64 (B) BF16 tiles into
// shared memory with TMA (128-byte swizzle) through a ring of mbarriers; warp 1 issues tcgen05.mma
// (M = 128, N = BN, K = 16 per instruction) from one thread into one of two tensor-memory
// accumulators (128 lanes x BN FP32 columns); warps 2 .. 9 read the other accumulator back and
// write the tile through shared memory, 64 consecutive columns of a row per store instruction.
// With one tile per CTA and four epilogue warps the wide product of the surrogate's reconstruction
// (40,000 x 16,834 x 384, 2.69 GB out) waited on loads, MMAs and stores in turn: 1.89 ms.
//
// Every wait is bounded (about a second of clock cycles); a wait that gives up sets
// kFlagTimeout in the caller's status word, the CTA stops issuing work, waits (bounded) for
// its own copies and MMAs in flight, frees its tensor memory and exits.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>

#include <type_traits>

#include "soap_internal.cuh"

namespace soap {
namespace tc {

constexpr int BM = 128;        // rows per CTA (TMEM lanes)
constexpr int BK = 64;         // K elements per stage: one 128-byte swizzle atom of BF16
constexpr int kEpiWarps = 8;   // two column halves of each group of 32 accumulator lanes
constexpr int kThreads = 64 + 32 * kEpiWarps;
template <int BN> struct Stages { static constexpr int value = BN >= 256 ? 3 : (BN >= 128 ? 4 : 6); };

struct Epilogue {
    const float* bias;          // [N] or NULL
    int gelu;
    float* c; int64_t ldc;
};

__device__ __forceinline__ float gelu(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float z) {
    // d/dz [z Phi(z)] = Phi(z) + z phi(z)
    return 0.5f * (1.0f + erff(z * 0.70710678118654752f)) + z * 0.39894228040143268f * __expf(-0.5f * z * z);
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ bool mbar_test(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait for the phase of parity `parity` to complete; false (and the flag) on timeout.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, unsigned int* flags) {
    const long long t0 = clock64();
    while (!mbar_test(bar, parity)) {
        if (clock64() - t0 > (1ll << 31)) {
            atomicOr(flags, kFlagTimeout);
            return false;
        }
    }
    return true;
}

__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, int c0, int c1, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(smem_u32(bar))
        : "memory");
}

// Shared-memory matrix descriptor: K-major operand, 128-byte swizzle, 8-row groups 1024 bytes
// apart (stride byte offset), descriptor version 1.
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFF);          // start address
    d |= (uint64_t)1 << 16;                          // leading byte offset (unused with swizzle)
    d |= (uint64_t)(1024 >> 4) << 32;                // stride byte offset
    d |= (uint64_t)1 << 46;                          // version
    d |= (uint64_t)2 << 61;                          // 128-byte swizzle
    return d;
}

// Instruction descriptor, kind::f16: FP32 accumulate, BF16 A and B, both K-major, M = 128.
__host__ __device__ constexpr uint32_t idesc_bf16(int n) {
    return (1u << 4)                       // D format FP32
           | (1u << 7)                     // A format BF16
           | (1u << 10)                    // B format BF16
           | ((uint32_t)(n >> 3) << 17)    // N / 8
           | ((uint32_t)(BM >> 4) << 24);  // M / 16
}

__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(tmem_d), "l"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
}

__device__ __forceinline__ void mma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                 ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; i++) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; i++) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float (&v)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%16], "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15};"
        ::"r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])), "r"(__float_as_uint(v[3])),
          "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])), "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7])),
          "r"(__float_as_uint(v[8])), "r"(__float_as_uint(v[9])), "r"(__float_as_uint(v[10])), "r"(__float_as_uint(v[11])),
          "r"(__float_as_uint(v[12])), "r"(__float_as_uint(v[13])), "r"(__float_as_uint(v[14])), "r"(__float_as_uint(v[15])),
          "r"(taddr)
        : "memory");
}

template <int BN>
struct Smem {
    static constexpr int STAGES = Stages<BN>::value;
    static constexpr int kA = BM * BK * 2;          // bytes per stage
    static constexpr int kB = BN * BK * 2;
    static constexpr int kStage = kA + kB;
    static constexpr int kCols = BN / 2 < 64 ? BN / 2 : 64;       // columns an epilogue warp stages at a time
    static constexpr int kPitch = kCols + 2;        // floats: 8-byte pairs of 16 rows fall on distinct banks
    static constexpr int kTile = 32 * kPitch * 4;
    static constexpr int kBytes = STAGES * kStage + kEpiWarps * kTile + 1024 /* alignment slack */ + 256 /* barriers */;
    static_assert(kBytes <= 227 * 1024, "shared memory of one CTA");
};

// Row-major store of a warp's 32 x 32 block through its shared tile: lane r holds row r's 32
// values; after the transpose, lane j writes column j of each row in turn, so every store
// instruction covers 32 consecutive elements of one row.
__device__ __forceinline__ void store_rows(float (*tile)[33], const float (&v)[32], int lane, float* base, int64_t ld,
                                           int m_first, int M, int n_first, int N) {
#pragma unroll
    for (int i = 0; i < 32; i++) tile[lane][i] = v[i];
    __syncwarp();
    const int n = n_first + lane;
    if (n < N) {
#pragma unroll 4
        for (int r = 0; r < 32; r++) {
            const int m = m_first + r;
            if (m >= M) break;
            base[(int64_t)m * ld + n] = tile[r][lane];
        }
    }
    __syncwarp();
}

// 40,000 x 16,834 x 384 (2.69 GB out): about 0.66 ms, 4.1 TB/s.  What bounds it there is the SM's
// shared-memory path: per 128 x 256 tile the MMAs read 288 KB of operands, the copies fill as much,
// and the output passes in and out (about 8,700 cycles at 128 bytes a cycle, of 9,100 measured;
// HBM alone would allow 6,100).
template <int BN>
__global__ void __launch_bounds__(kThreads, 1)
k_gemm_tn(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b, int M, int N,
          int K, Epilogue ep, unsigned int* flags) {
    static_assert(BN % 64 == 0 && BN <= 256, "tcgen05 N for M = 128, two accumulators in 512 columns");
    using SM = Smem<BN>;
    constexpr int STAGES = SM::STAGES;
    extern __shared__ unsigned char smem_raw[];
    // 1024-byte aligned operand ring (the swizzle atom), epilogue tiles and barriers after it
    unsigned char* ring = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    unsigned char* tiles = ring + STAGES * SM::kStage;
    uint64_t* full = reinterpret_cast<uint64_t*>(tiles + kEpiWarps * SM::kTile);
    uint64_t* empty = full + STAGES;
    uint64_t* acc_full = empty + STAGES;               // [2] accumulator complete
    uint64_t* acc_free = acc_full + 2;                 // [2] accumulator read back
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_free + 2);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n_kb = (K + BK - 1) / BK;
    const int tiles_n = (N + BN - 1) / BN;
    const int64_t n_tiles = (int64_t)((M + BM - 1) / BM) * tiles_n;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; s++) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
        for (int b = 0; b < 2; b++) { mbar_init(&acc_full[b], 1); mbar_init(&acc_free[b], kEpiWarps); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(tmem_slot)), "r"(2 * BN) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;

    if (warp == 0 && lane == 0) {
        // producer: it counts K blocks over all of this CTA's tiles
        int64_t it = 0;
        bool ok = true;
        for (int64_t tile = blockIdx.x; tile < n_tiles && ok; tile += gridDim.x) {
            const int m0 = (int)(tile / tiles_n) * BM, n0 = (int)(tile % tiles_n) * BN;
            for (int kb = 0; kb < n_kb; kb++, it++) {
                const int s = (int)(it % STAGES);
                if (!mbar_wait(&empty[s], (uint32_t)((it / STAGES) & 1) ^ 1, flags)) { ok = false; break; }
                unsigned char* a = ring + s * SM::kStage;
                mbar_expect_tx(&full[s], SM::kStage);
                tma_load_2d(a, &map_a, kb * BK, m0, &full[s]);
                tma_load_2d(a + SM::kA, &map_b, kb * BK, n0, &full[s]);
            }
        }
        // the last copies issued must land before the CTA may exit
        for (int64_t k = it - 1; k >= 0 && k >= it - STAGES; k--)
            mbar_wait(&full[k % STAGES], (uint32_t)((k / STAGES) & 1), flags);
    } else if (warp == 1 && lane == 0) {
        // MMA issuer
        constexpr uint32_t idesc = idesc_bf16(BN);
        int64_t it = 0;
        int n = 0;                                     // tiles so far
        bool ok = true;
        for (int64_t tile = blockIdx.x; tile < n_tiles && ok; tile += gridDim.x, n++) {
            const int buf = n & 1;
            if (!mbar_wait(&acc_free[buf], (uint32_t)((n >> 1) & 1) ^ 1, flags)) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            for (int kb = 0; kb < n_kb; kb++, it++) {
                const int s = (int)(it % STAGES);
                if (!mbar_wait(&full[s], (uint32_t)((it / STAGES) & 1), flags)) { ok = false; break; }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t a = smem_u32(ring + s * SM::kStage);
                const uint32_t b = a + SM::kA;
#pragma unroll
                for (int k = 0; k < BK / 16; k++)
                    mma_bf16(tmem + (uint32_t)(buf * BN), sdesc(a + k * 32), sdesc(b + k * 32), idesc, (kb | k) != 0);
                mma_commit(&empty[s]);
            }
            mma_commit(&acc_full[buf]);                // arrives once every MMA issued above has completed
        }
        // (bounded) every MMA has completed before the tensor memory can be released
        for (int k = n - 1; k >= 0 && k >= n - 2; k--) mbar_wait(&acc_full[k & 1], (uint32_t)((k >> 1) & 1), flags);
    } else if (warp >= 2) {
        // epilogue: TMEM lanes 32 (warp % 4) .. +31, columns of one half of the tile.  Lane r holds
        // row r's values; staged through the warp's tile, the lanes then run along the columns.
        constexpr int C = SM::kCols;
        const int lg = warp & 3, half = (warp - 2) >> 2;
        float* mine = reinterpret_cast<float*>(tiles + (warp - 2) * SM::kTile);
        const bool vec2 = (ep.ldc & 1) == 0 && (reinterpret_cast<uintptr_t>(ep.c) & 7) == 0;
        int n = 0;
        for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x, n++) {
            const int buf = n & 1;
            const int m0 = (int)(tile / tiles_n) * BM + 32 * lg, n0 = (int)(tile % tiles_n) * BN + half * (BN / 2);
            // warp-uniform decision: tcgen05.ld is a warp-wide (.sync.aligned) instruction
            if (!__all_sync(0xffffffffu, mbar_wait(&acc_full[buf], (uint32_t)((n >> 1) & 1), flags))) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t src = tmem + ((uint32_t)(32 * lg) << 16) + (uint32_t)(buf * BN + half * (BN / 2));
#pragma unroll 1
            for (int c = 0; c < BN / 2; c += C) {
#pragma unroll
                for (int q = 0; q < C; q += 32) {
                    float v[32];
                    tmem_ld32(src + (uint32_t)(c + q), v);
#pragma unroll
                    for (int i = 0; i < 16; i++)
                        *reinterpret_cast<float2*>(mine + lane * SM::kPitch + q + 2 * i) = make_float2(v[2 * i], v[2 * i + 1]);
                }
                if (c + C >= BN / 2) {                 // the accumulator is read: the next tile's MMAs may have it
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    __syncwarp();
                    if (lane == 0)
                        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&acc_free[buf])) : "memory");
                }
                __syncwarp();
                const int rows = min(32, M - m0), cols = min(C, N - n0 - c);
                float* dst = ep.c + (int64_t)m0 * ep.ldc + n0 + c;
                if (C == 64 && vec2 && rows == 32 && cols == 64) {
                    // whole block: sixteen rows in flight, no branches
                    const int j = 2 * lane;
                    const float2 b = ep.bias ? make_float2(__ldg(ep.bias + n0 + c + j), __ldg(ep.bias + n0 + c + j + 1))
                                             : make_float2(0.0f, 0.0f);
                    float* d = dst + j;
                    auto half_block = [&](int r0, auto with_bias, auto with_gelu) {
                        float2 x[16];
#pragma unroll
                        for (int r = 0; r < 16; r++)
                            x[r] = *reinterpret_cast<const float2*>(mine + (r0 + r) * SM::kPitch + j);
#pragma unroll
                        for (int r = 0; r < 16; r++) {
                            if (with_bias) { x[r].x += b.x; x[r].y += b.y; }
                            if (with_gelu) { x[r].x = gelu(x[r].x); x[r].y = gelu(x[r].y); }
                            *reinterpret_cast<float2*>(d) = x[r];
                            d += ep.ldc;
                        }
                    };
                    const bool hb = ep.bias != nullptr;
                    if (ep.gelu) { half_block(0, hb, true); half_block(16, hb, true); }
                    else if (hb) { half_block(0, std::true_type{}, std::false_type{}); half_block(16, std::true_type{}, std::false_type{}); }
                    else { half_block(0, std::false_type{}, std::false_type{}); half_block(16, std::false_type{}, std::false_type{}); }
                } else if (C == 64 && vec2) {
                    const int j = 2 * lane;
                    const float b0 = ep.bias && j < cols ? __ldg(ep.bias + n0 + c + j) : 0.0f;
                    const float b1 = ep.bias && j + 1 < cols ? __ldg(ep.bias + n0 + c + j + 1) : 0.0f;
#pragma unroll 8
                    for (int r = 0; r < rows; r++, dst += ep.ldc) {
                        float2 x = *reinterpret_cast<const float2*>(mine + r * SM::kPitch + j);
                        if (ep.bias) { x.x += b0; x.y += b1; }
                        if (ep.gelu) { x.x = gelu(x.x); x.y = gelu(x.y); }
                        if (j + 1 < cols) *reinterpret_cast<float2*>(dst + j) = x;
                        else if (j < cols) dst[j] = x.x;
                    }
                } else {
#pragma unroll 1
                    for (int j = lane; j < cols; j += 32) {
                        const float b0 = ep.bias ? __ldg(ep.bias + n0 + c + j) : 0.0f;
                        float* d = dst + j;
#pragma unroll 4
                        for (int r = 0; r < rows; r++, d += ep.ldc) {
                            float x = mine[r * SM::kPitch + j];
                            if (ep.bias) x += b0;
                            *d = ep.gelu ? gelu(x) : x;
                        }
                    }
                }
                __syncwarp();
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * BN) : "memory");
    }
}

// Row-major BF16 matrix [rows][cols] with row stride ld (elements): boxes of box_rows x 64, 128-byte
// swizzle, zero fill outside.
soap_status operand_map(CUtensorMap* map, const void* base, int64_t rows, int64_t cols, int64_t ld, int box_rows);

// Tiled tensor map without swizzle (BF16 elements unless dt says otherwise): dims[0] innermost
// (elements), strides in bytes of dims 1 .. rank-1, box in elements.  Zero fill outside the tensor.
soap_status encode_map(CUtensorMap* map, int rank, const void* base, const uint64_t* dims,
                       const uint64_t* strides, const uint32_t* box,
                       CUtensorMapDataType dt = CU_TENSOR_MAP_DATA_TYPE_BFLOAT16);

// C = act(A B^T + bias): A [M][K] (row stride lda), B [N][K] (row stride ldb), BF16, device, with
// 16-byte aligned bases and strides that are multiples of 8 elements.  Asynchronous on `st`.
soap_status gemm_tn(const __nv_bfloat16* A, int64_t lda, const __nv_bfloat16* B, int64_t ldb, int M, int N,
                    int K, const Epilogue& ep, cudaStream_t st, unsigned int* flags);

}  // namespace tc
}  // namespace soap

// pca_tc.cu -- projection of spectra onto a PCA basis, coef = (X - mean) basis^T, on the tensor
// cores at FP32 accuracy.
//
// An FP32 number is exactly the sum of three BF16 numbers (8 significant bits each): x = h + m + l.
// Of the nine products of two such sums, six (hh, hm, mh, hl, lh, mm) are computed; the dropped
// ones are below 2^-24 of the product, FP32's own rounding.  The tensor cores add into FP32
// accumulators; hh has one of its own, and every kDrain blocks of 64 pixels they are added, the
// small products first, to a running FP32 sum, so that neither a long chain of additions nor the
// accumulator's rounding costs accuracy (against float64 on 20,011 x 16,834 x 128 normal values:
// 4.9e-7 of the norm; the FP32 product summed in order 2.8e-6).
//
// k_project: one persistent CTA per SM; the work is (tiles of 128 rows x 128 components) x (blocks
// of 64 pixels), cut evenly between the CTAs wherever that falls inside a tile, so that 157 tiles
// do not take two rounds on 152 SMs.  A tile is cut at most once: its two partial sums are added
// to a cleared output, and 0 + a + b is the same in either order.  Per block sixteen warps load 128
// rows of X and of the basis (lanes along the pixels: coalesced for any alignment), subtract the
// mean, split and store both operands as 128-byte-swizzled K-major tiles.  Four more warps: a lane
// of the first issues the MMAs, all four drain the accumulators.  The running sums live in tensor
// memory: in registers (of the splitters or of warps of their own) they made the splitters' prefetch
// spill, and a spilled value waits for its load (the call below 763 us with 20 bytes spilled, 1,110 with 260).
// 20,011 x 16,834 x 128: 0.57 ms a call (2.4 TB/s of X), against 5.5 ms as an FP32 SIMT product of
// 64 x 64 tiles and a product of one row (the mean) on two SMs; without the loads it takes 0.45, and
// without the MMAs 0.47: splitting (about eleven instructions per pixel pair and operand) and the
// shared memory that splits, loads and MMAs share bound it.
//
// Waits are bounded as in tc_gemm.cuh.
#include <algorithm>
#include <cmath>

#include "tc_gemm.cuh"

namespace soap {
namespace pca {

constexpr int kTile = 128;                             // rows and components per tile
constexpr int kPart = kTile * 128;                     // one split part of one operand block, bytes
constexpr int kStage = 6 * kPart;                      // A h, m, l and B h, m, l
constexpr int kStages = 2;
constexpr int kSplitWarps = 16;
constexpr int kRows = kTile / kSplitWarps;             // rows of each operand a warp splits
constexpr int kThreads = 32 * (kSplitWarps + 4);
constexpr int kDrain = 8;
constexpr int kSmem = kStages * kStage + 1024 + 256;

struct Args {
    const float* x;            // [n][p]
    const float* mean;         // [p]
    const float* basis;        // [k][p]
    float* coef;               // [n][k]
    int64_t n, p;
    int k, tiles_k;
    int blocks;                // 64-pixel blocks per tile
    int units, per_cta;        // tile blocks in all, and per CTA (0: two CTAs per tile)
};

// Loads of the next block's values, issued a block ahead.  Volatile: the compiler would otherwise
// sink a read-only load past the waits to its use, which undoes the prefetch.
__device__ __forceinline__ float ld1(const float* p) {
    float v;
    asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ float2 ld2(const float* p) {
    float2 v;
    asm volatile("ld.global.nc.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
    return v;
}

// Two pixels of kRows rows, `left` rows following the first; past the end the last row repeats (those
// rows and components are not stored).  `past`: how far the pair reaches past the row's last pixel:
// it is moved back, or its second pixel is, and zeroed in the split.
template <bool kVec>
__device__ __forceinline__ void load_rows(float2 (&v)[kRows], const float* src, int64_t p, int left, int past) {
    int second = 1;
    if (past > 0) {
        src -= kVec ? past : past - 1;
        second = 0;
    }
#pragma unroll
    for (int i = 0; i < kRows; i++) {
        if constexpr (kVec) v[i] = ld2(src);
        else v[i] = make_float2(ld1(src), ld1(src + second));
        if (i < left) src += p;
    }
}

__device__ __forceinline__ uint32_t top(float a, float b, float& ra, float& rb) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    const float2 f = __bfloat1622float2(h);
    ra = a - f.x;
    rb = b - f.y;
    return *reinterpret_cast<const uint32_t*>(&h);
}

// the three parts of a pixel pair into the operand's three tiles
__device__ __forceinline__ void put(unsigned char* part, uint32_t off, float2 v) {
    float a, b, c, d;
    *reinterpret_cast<uint32_t*>(part + off) = top(v.x, v.y, a, b);
    *reinterpret_cast<uint32_t*>(part + kPart + off) = top(a, b, c, d);
    *reinterpret_cast<uint32_t*>(part + 2 * kPart + off) = top(c, d, a, b);
}

template <bool kVec>
__global__ void __launch_bounds__(kThreads, 1)
k_project(const __grid_constant__ Args g, unsigned int* flags) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char* ring = smem_raw + ((1024u - (tc::smem_u32(smem_raw) & 1023u)) & 1023u);
    uint64_t* full = reinterpret_cast<uint64_t*>(ring + kStages * kStage);
    uint64_t* empty = full + kStages;
    uint64_t* acc_full = empty + kStages;
    uint64_t* acc_free = acc_full + 1;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_free + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int u0 = (int)blockIdx.x * g.per_cta, u1 = min(g.units, u0 + g.per_cta);
    if (g.per_cta == 0) {
        const int tile0 = (int)(blockIdx.x >> 1) * g.blocks, mid = tile0 + (g.blocks + 1) / 2;
        u0 = blockIdx.x & 1 ? mid : tile0;
        u1 = blockIdx.x & 1 ? tile0 + g.blocks : mid;
    }

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; s++) { tc::mbar_init(&full[s], 32 * kSplitWarps); tc::mbar_init(&empty[s], 1); }
        tc::mbar_init(acc_full, 1);
        tc::mbar_init(acc_free, 128);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(tc::smem_u32(tmem_slot)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;                  // columns 0: hh; 128: hm, hl, mh, lh; 256: mm; 384: sums

    if (warp < kSplitWarps) {
        // splitters: warp w takes rows 8 w .. of both operands
        const int r0 = kRows * warp;
        float2 a[kRows], b[kRows], mu;
        // the block to load next: its tile, this lane's pixels in the warp's first rows, rows left
        int tile = u0 / g.blocks, blk = u0 - tile * g.blocks, left_a, left_b;
        const float *pa, *pb, *pm;
        auto at_tile = [&]() {
            const int64_t row = (int64_t)(tile / g.tiles_k) * kTile + r0;
            const int comp = tile % g.tiles_k * kTile + r0;
            const int64_t ra = row < g.n ? row : g.n - 1, px = 64ll * blk + 2 * lane;
            const int rb = min(comp, g.k - 1);
            left_a = (int)min((int64_t)kRows, g.n - 1 - ra);
            left_b = min(kRows, g.k - 1 - rb);
            pa = g.x + ra * g.p + px;
            pb = g.basis + rb * g.p + px;
            pm = g.mean + px;
        };
        auto advance = [&]() {
            if (++blk < g.blocks) {
                pa += 64;
                pb += 64;
                pm += 64;
            } else {
                blk = 0;
                tile++;
                at_tile();
            }
        };
        // how far the pair of block blk reaches past the row
        auto past = [&]() { return blk + 1 < g.blocks ? 0 : max(0, (int)(64ll * blk + 2 * lane + 2 - g.p)); };
        auto load_a = [&]() {
            const int over = past();
            load_rows<kVec>(a, pa, g.p, left_a, over);
            mu.x = ld1(pm - max(0, over - 1));
            mu.y = ld1(pm + 1 - over);
        };
        auto load_b = [&]() { load_rows<kVec>(b, pb, g.p, left_b, past()); };
        at_tile();
        if (u0 < u1) { load_a(); load_b(); }
        // this lane's place in row r of a swizzled tile: by r mod 8
        const uint32_t lane_off = (uint32_t)(4 * (lane & 3));
        for (int u = u0, it = 0; u < u1; u++, it++) {
            const int s = it % kStages;
            if (!tc::mbar_wait(&empty[s], (uint32_t)((it / kStages) & 1) ^ 1, flags)) break;
            unsigned char* st = ring + s * kStage + r0 * 128;
            const int over = past();
            if (over > 0) {
#pragma unroll
                for (int i = 0; i < kRows; i++) {
                    if (over > 1) { a[i].x = mu.x; b[i].x = 0.0f; }
                    a[i].y = mu.y;
                    b[i].y = 0.0f;
                }
            }
            advance();
#pragma unroll
            for (int i = 0; i < kRows; i++)
                put(st, (uint32_t)(i * 128) + lane_off + (uint32_t)(((lane >> 2) ^ (i & 7)) << 4),
                    make_float2(a[i].x - mu.x, a[i].y - mu.y));
            if (u + 1 < u1) load_a();
#pragma unroll
            for (int i = 0; i < kRows; i++)
                put(st + 3 * kPart, (uint32_t)(i * 128) + lane_off + (uint32_t)(((lane >> 2) ^ (i & 7)) << 4), b[i]);
            if (u + 1 < u1) load_b();
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");     // visible to the tensor cores
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_u32(&full[s])) : "memory");
        }
    } else {
        const int lg = warp & 3;
        const uint32_t src = tmem + ((uint32_t)(32 * lg) << 16);
        int it = 0, groups = 0;                        // blocks, accumulator groups so far
        bool ok = true;
        for (int u = u0; u < u1 && ok;) {
            const int tile = u / g.blocks, begin = u, end = min(u1, (tile + 1) * g.blocks);
            for (; u < end; groups++) {                // blocks of one tile, kDrain to a group
                const int stop = min(end, u + kDrain);
                if (warp == kSplitWarps && lane == 0) {
                    ok = groups == 0 || tc::mbar_wait(acc_free, (uint32_t)((groups - 1) & 1), flags);
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    // B's h and m tiles lie one after the other: as one operand of 256 columns they
                    // halve what the MMAs read of A for those products
                    constexpr uint32_t one = tc::idesc_bf16(kTile), two = tc::idesc_bf16(2 * kTile);
                    for (int v = u; v < stop && ok; v++, it++) {
                        const int s = it % kStages;
                        if (!tc::mbar_wait(&full[s], (uint32_t)((it / kStages) & 1), flags)) { ok = false; break; }
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        const uint32_t ah = tc::smem_u32(ring + s * kStage), am = ah + kPart, al = am + kPart;
                        const uint32_t bh = al + kPart, bl = bh + 2 * kPart;
#pragma unroll
                        for (int q = 0; q < 4; q++) {
                            const uint32_t o = 32 * q, acc = v > u || q;
                            tc::mma_bf16(tmem, tc::sdesc(ah + o), tc::sdesc(bh + o), two, acc);           // hh | hm
                            if (!acc) {                // (the third accumulator starts at zero too)
                                tc::mma_bf16(tmem + 128u, tc::sdesc(am + o), tc::sdesc(bh + o), one, 1u);
                                tc::mma_bf16(tmem + 256u, tc::sdesc(am + o), tc::sdesc(bh + kPart + o), one, 0u);
                            } else {
                                tc::mma_bf16(tmem + 128u, tc::sdesc(am + o), tc::sdesc(bh + o), two, 1u); // mh | mm
                            }
                            tc::mma_bf16(tmem + 128u, tc::sdesc(ah + o), tc::sdesc(bl + o), one, 1u);
                            tc::mma_bf16(tmem + 128u, tc::sdesc(al + o), tc::sdesc(bh + o), one, 1u);
                        }
                        tc::mma_commit(&empty[s]);
                    }
                    tc::mma_commit(acc_full);          // arrives once every MMA issued above has completed
                }
                const bool first = u == begin;
                u = stop;
                ok = __all_sync(0xffffffffu, tc::mbar_wait(acc_full, (uint32_t)(groups & 1), flags) && ok);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll 1
                for (int c = 0; c < kTile; c += 16) {
                    float sum[16], v[16];
#pragma unroll
                    for (int q = 3; q >= 0; q--) {     // the running sum, then the small products first
                        if (q == 3 && first) {
#pragma unroll
                            for (int i = 0; i < 16; i++) sum[i] = 0.0f;
                            continue;
                        }
                        tc::tmem_ld16(src + 128u * q + (uint32_t)c, v);
#pragma unroll
                        for (int i = 0; i < 16; i++) sum[i] = q == 3 ? v[i] : sum[i] + v[i];
                    }
                    tc::tmem_st16(src + 384u + (uint32_t)c, sum);
                }
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_u32(acc_free)) : "memory");
            }
            if (!ok) break;
            // the tile's sums: stored, or added when another CTA has the rest of the tile
            const int64_t row = (int64_t)(tile / g.tiles_k) * kTile + 32 * lg + lane;
            const int c0 = tile % g.tiles_k * kTile, cols = min(kTile, g.k - c0);
            const bool whole = end - begin == g.blocks;
            const bool vec4 = (g.k & 3) == 0 && (reinterpret_cast<uintptr_t>(g.coef) & 15) == 0;
#pragma unroll 1
            for (int c = 0; c < cols; c += 16) {
                float sum[16];
                tc::tmem_ld16(src + 384u + (uint32_t)c, sum);
                if (row < g.n) {
                    float* dst = g.coef + row * g.k + c0 + c;
                    if (whole && vec4 && c + 16 <= cols) {
#pragma unroll
                        for (int i = 0; i < 4; i++)
                            reinterpret_cast<float4*>(dst)[i] =
                                make_float4(sum[4 * i], sum[4 * i + 1], sum[4 * i + 2], sum[4 * i + 3]);
                    } else {
#pragma unroll
                        for (int i = 0; i < 16; i++)
                            if (c + i < cols) {
                                if (whole) dst[i] = sum[i];
                                else atomicAdd(dst + i, sum[i]);
                            }
                    }
                }
                __syncwarp();
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
}

// Coefficients that did not come out finite, again with plain FP32 products: an infinity (or a
// value that rounds to one in BF16) has no exact split, and times a zero part it would be a NaN
// where FP32 gives an infinity.  Warp per coefficient found; a pass over finite ones only reads.
__global__ void __launch_bounds__(256)
k_project_nonfinite(Args g) {
    const int64_t total = g.n * g.k;
    const int lane = threadIdx.x & 31;
    for (int64_t e0 = ((int64_t)blockIdx.x * 256 + threadIdx.x) / 32 * 32; e0 < total; e0 += (int64_t)gridDim.x * 256) {
        const int64_t e = e0 + lane;
        unsigned int bad = __ballot_sync(0xffffffffu, e < total && !isfinite(g.coef[e]));
        while (bad) {
            const int64_t q = e0 + __ffs(bad) - 1;
            bad &= bad - 1;
            const float* x = g.x + q / g.k * g.p;
            const float* v = g.basis + q % g.k * g.p;
            float s = 0.0f, m = 0.0f;
            for (int64_t i = lane; i < g.p; i += 32) {
                s = fmaf(x[i], v[i], s);
                m = fmaf(g.mean[i], v[i], m);
            }
            for (int o = 16; o > 0; o >>= 1) {
                s += __shfl_xor_sync(0xffffffffu, s, o);
                m += __shfl_xor_sync(0xffffffffu, m, o);
            }
            if (lane == 0) g.coef[q] = s - m;
        }
    }
}

soap_status project(const float* x, int64_t n, int64_t p, const float* mean, const float* basis, int k, float* coef,
                    cudaStream_t st) {
    int dev = 0, sms = 0;
    SOAP_CUDA(cudaGetDevice(&dev));
    SOAP_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    CallStatus status(st);
    unsigned int* flags = nullptr;
    SOAP_TRY(status.begin(&flags));
    Args a{};
    a.x = x; a.mean = mean; a.basis = basis; a.coef = coef;
    a.n = n; a.p = p; a.k = k;
    a.tiles_k = (k + kTile - 1) / kTile;
    const int64_t blocks = (p + 63) / 64, tiles = (n + kTile - 1) / kTile * a.tiles_k, units = tiles * blocks;
    if (units > INT32_MAX - 2 * blocks) { set_error("%lld x %lld spectra in one projection", (long long)n, (long long)p); return SOAP_ERANGE; }
    a.blocks = (int)blocks;
    a.units = (int)units;
    // Even shares of at least a tile (so that a tile is cut at most once), or two CTAs to each tile
    // while that many fit on the GPU.
    a.per_cta = 2 * tiles <= sms ? 0 : std::max(a.blocks, (a.units + sms - 1) / sms);
    const int ctas = a.per_cta ? (a.units + a.per_cta - 1) / a.per_cta : (int)(2 * tiles);
    if (a.per_cta != a.blocks) SOAP_CUDA(cudaMemsetAsync(coef, 0, (size_t)n * k * sizeof(float), st));
    const bool vec = p % 2 == 0 && (reinterpret_cast<uintptr_t>(x) & 7) == 0 && (reinterpret_cast<uintptr_t>(basis) & 7) == 0;
    if (vec) {                                         // pixel pairs in one load
        SOAP_TRY(fit_dynamic_smem(k_project<true>, kSmem));
        k_project<true><<<(unsigned)ctas, kThreads, kSmem, st>>>(a, flags);
    } else {
        SOAP_TRY(fit_dynamic_smem(k_project<false>, kSmem));
        k_project<false><<<(unsigned)ctas, kThreads, kSmem, st>>>(a, flags);
    }
    SOAP_CUDA(cudaGetLastError());
    k_project_nonfinite<<<(unsigned)std::min<int64_t>((n * k + 255) / 256, 8 * sms), 256, 0, st>>>(a);
    SOAP_CUDA(cudaGetLastError());
    unsigned int h = 0;
    SOAP_TRY(status.finish(&h));
    if (h) { set_error("the projection kernel gave up waiting (status 0x%x)", h); return SOAP_ETIMEOUT; }
    return SOAP_OK;
}

}  // namespace pca
}  // namespace soap

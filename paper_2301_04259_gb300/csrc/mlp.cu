// mlp.cu -- the surrogate network's layers chained inside one kernel, forward (queries) and
// forward + loss + backward (training), and the weight gradients of a batch in one launch.
//
// k_mlp: a CTA owns 128 rows through every layer.  The rows' BF16 activations live in shared
// memory as the K-major A operand of the next product (4 swizzle atoms of 128 rows x 64 columns),
// the accumulator in tensor memory; only weights are streamed (64-column K blocks of 256 rows
// through a ring of 4 TMA stages, which run ahead of the layer being computed).
//   warp 0, one lane    weight copies
//   warp 1, one lane    the MMAs (M = 128, N = 256 or 144, K = 16), and in training the TMA stores
//                       of the activations / gradients straight out of the operand buffer
//   warps 2 .. 17       epilogues: warp w reads TMEM lanes 32 (w mod 4) .., 64 columns of the
//                       layer, i.e. one swizzle atom of the next operand
// What bounds it is the epilogue's arithmetic (erff and the exponential of GELU'), so sixteen warps
// share it, and GELU'(z) is taken in the forward pass, where erff(z / sqrt 2) is at hand anyway.
// A training step with too few rows for every SM (kPair): a cluster of two CTAs shares 128 rows.  Each
// computes half of a hidden layer's columns, with half the weights and half the epilogue, and copies its half of the next
// operand into the other's buffer (shared memory to shared memory, counted on the receiver's barrier).
// The accumulator barriers count the MMAs of both, so a half is only overwritten when both products
// that read it are complete.  The inputs, the output layer and its gradient are computed by both.
// 4,096 rows: 68 us in 64 CTAs, 76 in 32 (16 such steps with their gradients and Adam 1,918 -> 1,777 us);
// with a layer's biases, and the GELU' factors of the backward products, fetched while the product is
// computed 65 (1,753).
// Not for queries: 7 of them took 28 us instead of 34, which their call did not show.
// As one kernel per layer a tile's epilogue ran on four warps (28 us a 128 x 256 layer) and every
// activation went through global memory twice, row-major and transposed: a training step of 4,096
// rows took 18 launches and 0.65 ms, 7 queries 345 us (see surrogate.cu for the times now).
//
// k_mlp_dw: dW_l = g_l^T a_{l-1} for all layers at once, one CTA per 128 x 64 tile, K = the whole
// batch in order (as one chain of MMAs, so the sums do not depend on the tiling).  Both operands
// are row-major over the batch, i.e. MN-major for this product, which the tensor cores read as
// stored; so no transposed copies are written.  The launch's last blocks take the bias gradients.
//
// Waits are bounded as in tc_gemm.cuh.
#include "mlp.cuh"

#include <cfloat>

using bf16 = __nv_bfloat16;

namespace soap {
namespace mlp {

constexpr int kRows = 128;
constexpr int kAtom = kRows * 128;                     // one operand atom: 128 rows x 128 bytes
constexpr int kActBytes = 4 * kAtom;
constexpr int kWStage = kHidden * 128;                 // one K block of weights: 256 rows x 128 bytes
constexpr int kWStages = 4;
constexpr int kEpiWarps = 16;
constexpr int kThreads = 64 + 32 * kEpiWarps;
constexpr int kSmem = kActBytes + kWStages * kWStage + 1024 + 256;
static_assert(kEpiWarps * 32 * 33 * 4 <= kWStages * kWStage, "the coefficient tiles reuse the weight ring");

__device__ __forceinline__ float scale_in(float x, float lo, float hi) { return 2.0f * (x - lo) / (hi - lo) - 1.0f; }

// volatile: the compiler would otherwise sink a read-only load past the wait to its use
__device__ __forceinline__ float4 ld4(const float4* p) {
    float4 v;
    asm volatile("ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
    return v;
}

__device__ __forceinline__ uint32_t pack2(float a, float b) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&h);
}

// 32 values of one row, columns 32 h .. of an operand atom, as four swizzled 16-byte chunks
__device__ __forceinline__ void put_row(unsigned char* atom, int r, int h, const float (&a)[32]) {
#pragma unroll
    for (int j = 0; j < 4; j++) {
        const uint4 v = make_uint4(pack2(a[8 * j], a[8 * j + 1]), pack2(a[8 * j + 2], a[8 * j + 3]),
                                   pack2(a[8 * j + 4], a[8 * j + 5]), pack2(a[8 * j + 6], a[8 * j + 7]));
        *reinterpret_cast<uint4*>(atom + r * 128 + (((4 * h + j) ^ (r & 7)) << 4)) = v;
    }
}

__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, const void* src, int c0, int c1) {
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];"
                 ::"l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(tc::smem_u32(src)) : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_u32(bar)) : "memory");
}

// the operand buffer's first n_atoms atoms to rows row0 .. of a row-major matrix (columns past its
// width are clipped); kPair: this CTA's two of them
template <bool kPair>
__device__ __forceinline__ void store_operand(const CUtensorMap* map, const unsigned char* act, int n_atoms, int row0,
                                              uint32_t rank) {
    for (int q = kPair ? 2 * (int)rank : 0; q < (kPair ? 2 * (int)rank + 2 : n_atoms); q++)
        for (int h = 0; h < 2; h++) tma_store_2d(map, act + q * kAtom + h * (kAtom / 2), 64 * q, row0 + 64 * h);
    bulk_commit();
}

__device__ __forceinline__ uint32_t peer_addr(const void* p, uint32_t rank) {
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(tc::smem_u32(p)), "r"(rank));
    return a;
}
// the same place of the other CTA's shared memory, its barrier counting the bytes
__device__ __forceinline__ void copy_to_peer(const void* src, uint32_t bytes, const uint64_t* bar, uint32_t peer) {
    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(peer_addr(src, peer)), "r"(tc::smem_u32(src)), "r"(bytes), "r"(peer_addr(bar, peer)) : "memory");
}
__device__ __forceinline__ void commit_both(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 ::"r"(tc::smem_u32(bar)), "h"((uint16_t)3) : "memory");
}
__device__ __forceinline__ void pair_sync() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

__host__ __device__ constexpr int k_blocks(int q) { return q == 0 ? 1 : (q == 5 ? 3 : 4); }

// product q: 0 .. 4 forward, 5 .. 8 backward
template <bool kTrain, bool kPair>
__device__ __forceinline__ void chain(const Weights& w, const TrainArgs* ta, const QueryArgs* qa, int64_t row0,
                                      unsigned int* flags) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char* act = smem_raw + ((1024u - (tc::smem_u32(smem_raw) & 1023u)) & 1023u);
    unsigned char* ring = act + kActBytes;
    uint64_t* full = reinterpret_cast<uint64_t*>(ring + kWStages * kWStage);
    uint64_t* empty = full + kWStages;
    uint64_t* ready = empty + kWStages;                // the operand buffer holds the next product's A
    uint64_t* accum = ready + 1;
    uint64_t* theirs = accum + 1;                      // kPair: the other's half of the operand has landed
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(theirs + 1);
    const uint32_t rank = kPair ? blockIdx.x & 1u : 0u;
    constexpr int kHalf = kHidden / 2;
    constexpr int kProducts = kTrain ? kFwd + kBwd : kFwd;
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;

    if (t == 0) {
        for (int s = 0; s < kWStages; s++) { tc::mbar_init(&full[s], 1); tc::mbar_init(&empty[s], 1); }
        tc::mbar_init(ready, 32 * kEpiWarps);
        tc::mbar_init(accum, kPair ? 2 : 1);
        tc::mbar_init(theirs, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(tc::smem_u32(tmem_slot)), "r"(256) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if constexpr (kPair) pair_sync();                  // the other's barriers exist before anything arrives there
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        if (lane == 0) {
            int it = 0;
            bool ok = true;
            for (int q = 0; q < kProducts && ok; q++) {
                const CUtensorMap* map = q < kFwd ? &w.fwd[q] : &w.bwd[q - kFwd];
                for (int kb = 0; kb < k_blocks(q); kb++) {
                    const int s = it % kWStages;
                    if (!tc::mbar_wait(&empty[s], ((it / kWStages) & 1) ^ 1, flags)) { ok = false; break; }
                    // 128 outputs a copy: this CTA's half of a hidden layer's, or both
                    const bool half = kPair && q != kFwd - 1;
                    tc::mbar_expect_tx(&full[s], half ? kWStage / 2 : kWStage);
                    tc::tma_load_2d(ring + s * kWStage, map, kb * 64, half ? (int)rank * kHalf : 0, &full[s]);
                    if (!half) tc::tma_load_2d(ring + s * kWStage + kWStage / 2, map, kb * 64, kHalf, &full[s]);
                    it++;
                }
            }
            // the last copies issued must land before the CTA may exit
            for (int k = it - 1; k >= 0 && k >= it - kWStages; k--)
                tc::mbar_wait(&full[k % kWStages], (k / kWStages) & 1, flags);
        }
    } else if (warp == 1) {
        if (lane == 0) {
            int it = 0, exchanges = 0;
            bool ok = true;
            for (int q = 0; q < kProducts && ok; q++) {
                if (!tc::mbar_wait(ready, q & 1, flags)) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                // operands that the epilogues of both wrote a half of: this half to the other (whose
                // products on the operand before are complete, as the epilogue waited for them)
                const bool shared = kPair && q != 0 && q != kFwd;
                if (shared) {
                    tc::mbar_expect_tx(theirs, 2 * kAtom);
                    copy_to_peer(act + 2 * rank * kAtom, 2 * kAtom, theirs, rank ^ 1u);
                }
                if constexpr (kTrain) {                // what this product reads is also kept for dW
                    if (q >= 1 && q < kFwd) store_operand<kPair>(&ta->s.a[q], act, 4, (int)row0, rank);
                    else if (q == kFwd && rank == 0) store_operand<false>(&ta->s.g[4], act, 3, (int)row0, 0);
                    else if (q > kFwd) store_operand<kPair>(&ta->s.g[kFwd + kBwd - q], act, 4, (int)row0, rank);
                }
                const uint32_t idesc = tc::idesc_bf16(q == kFwd - 1 ? 144 : (kPair ? kHalf : 256));
                for (int kb = 0; kb < k_blocks(q) && ok; kb++, it++) {
                    const int s = it % kWStages;
                    if (shared && kb == (rank == 0 ? 2 : 0)) {
                        ok = tc::mbar_wait(theirs, exchanges & 1, flags);
                        exchanges++;
                        if (!ok) break;
                    }
                    if (!tc::mbar_wait(&full[s], (it / kWStages) & 1, flags)) { ok = false; break; }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t a = tc::smem_u32(act + kb * kAtom), b = tc::smem_u32(ring + s * kWStage);
                    const int nk = q == 0 ? 1 : 4;     // the first layer's 8 inputs fill half a K step
                    for (int k = 0; k < nk; k++)
                        tc::mma_bf16(tmem, tc::sdesc(a + k * 32), tc::sdesc(b + k * 32), idesc, (kb | k) != 0);
                    tc::mma_commit(&empty[s]);
                }
                // the epilogue overwrites the operand buffer: its stores must have read it
                if constexpr (kTrain) bulk_wait_read();
                // arrives once every MMA issued above has completed
                if constexpr (kPair) commit_both(accum);
                else tc::mma_commit(accum);
            }
            if constexpr (kTrain) {
                if (ok && tc::mbar_wait(ready, kProducts & 1, flags)) store_operand<kPair>(&ta->s.g[0], act, 4, (int)row0, rank);
                bulk_wait_all();
            }
        }
    } else {
        const int lg = warp & 3, qd = (warp - 2) >> 2;
        const int r = 32 * lg + lane;
        // epilogue thread: its place in the grad buffers
        const int grad0 = t - 64 + (int)rank * (32 * kEpiWarps * 8);
        const uint32_t tbase = tmem + ((uint32_t)(32 * lg) << 16);
        // a warp's columns of a hidden layer: 64, or 32 of this CTA's half
        constexpr int kCols = kPair ? 32 : 64;
        const int col0 = kPair ? kHalf * (int)rank + 32 * qd : 64 * qd;
        unsigned char* atom = act + (col0 / 64) * kAtom;
        auto publish = [&]() {
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // visible to the tensor cores and TMA
            mbar_arrive(ready);
        };
        int64_t src = row0 + r;
        const float* x;
        bool row_on = true;
        if constexpr (kTrain) {
            if (ta->perm) src = ta->perm[(int64_t)ta->d_step[0] * ta->B + row0 + r];
            x = ta->x;
        } else {
            row_on = src < qa->n;
            if (!row_on) src = qa->n - 1;
            x = qa->x;
        }
        const float* lohi = kTrain ? ta->lohi : qa->lohi;
        bool in_range = true;
        if (qd == 0 || (!kTrain && qd == 2)) {
            float v[kIn];
#pragma unroll
            for (int i = 0; i < kIn; i++) {
                const float xi = __ldg(x + src * kIn + i), lo = __ldg(lohi + i), hi = __ldg(lohi + kIn + i);
                in_range = in_range && xi >= lo && xi <= hi;
                v[i] = scale_in(xi, lo, hi);
            }
            if (qd == 0) {
                const uint4 c = make_uint4(pack2(v[0], v[1]), pack2(v[2], v[3]), pack2(v[4], v[5]), pack2(v[6], v[7]));
                *reinterpret_cast<uint4*>(act + r * 128 + ((r & 7) << 4)) = c;
                *reinterpret_cast<uint4*>(act + r * 128 + ((1 ^ (r & 7)) << 4)) = make_uint4(0, 0, 0, 0);
                if constexpr (kTrain)
                    if (rank == 0) *reinterpret_cast<uint4*>(ta->s.x0 + (row0 + r) * kIn) = c;
            }
        }
        publish();
        bool ok = true;
        // forward layers
        for (int l = 0; l < kFwd - 1 && ok; l++) {
            // the first 32 columns' biases are fetched while the product is computed
            const float4* bias = reinterpret_cast<const float4*>(w.bias[l] + col0);
            float4 b4[8];
#pragma unroll
            for (int j = 0; j < 8; j++) b4[j] = ld4(bias + j);
            ok = __all_sync(0xffffffffu, tc::mbar_wait(accum, l & 1, flags));
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            if (!ok) break;
#pragma unroll 1
            for (int h = 0; h < kCols / 32; h++) {
                if (h > 0) {
#pragma unroll
                    for (int j = 0; j < 8; j++) b4[j] = ld4(bias + 8 * h + j);
                }
                float v[32];
                tc::tmem_ld32(tbase + (uint32_t)(kCols * qd + 32 * h), v);
                float4* gr = kTrain ? reinterpret_cast<float4*>(ta->s.grad[l]) + row0 * (kHidden / 4) + grad0 : nullptr;
#pragma unroll
                for (int j = 0; j < 8; j++) {
                    const float z0 = v[4 * j] + b4[j].x, z1 = v[4 * j + 1] + b4[j].y, z2 = v[4 * j + 2] + b4[j].z,
                                z3 = v[4 * j + 3] + b4[j].w;
                    if constexpr (kTrain)
                        gr[(8 * h + j) * (32 * kEpiWarps)] =
                            make_float4(tc::gelu_grad(z0), tc::gelu_grad(z1), tc::gelu_grad(z2), tc::gelu_grad(z3));
                    v[4 * j] = tc::gelu(z0);
                    v[4 * j + 1] = tc::gelu(z1);
                    v[4 * j + 2] = tc::gelu(z2);
                    v[4 * j + 3] = tc::gelu(z3);
                }
                put_row(atom, r, kPair ? qd & 1 : h, v);
            }
            publish();
        }
        // outputs
        if (ok) {
            ok = __all_sync(0xffffffffu, tc::mbar_wait(accum, (kFwd - 1) & 1, flags));
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        }
        const float* bias = w.bias[kFwd - 1];
        if constexpr (kTrain) {
            // L = sum_b sum_j w_j (y - t)^2 / B, dL/dy = 2 w_j (y - t) / B.  A thread's part of L, which is
            // reported and enters no gradient, is a pair of floats (the rounding error of a product by an
            // FMA, of a sum by TwoSum): ~48 bits, five fewer than FP64's, without FP64 arithmetic, which
            // runs at 1/64 rate.  A warp whose squares or sums leave FP32's range takes them in FP64.
            if (ok && qd < 3) {
                float hi = 0.0f, lo = 0.0f;
                const float* trow = ta->t + src * kOut;
#pragma unroll 1
                for (int h = 0; h < 2; h++) {
                    const int c = 64 * qd + 32 * h;
                    float v[32];
                    if (c < kOutPad) tc::tmem_ld32(tbase + (uint32_t)c, v);
#pragma unroll
                    for (int i = 0; i < 32; i++) {
                        const int j = c + i;
                        if (j >= kOut) { v[i] = 0.0f; continue; }
                        const float res = v[i] + __ldg(bias + j) - __ldg(trow + j);
                        const float wj = __ldg(ta->w_out + j);
                        const float s = res * res, p = wj * s;
                        const float e = fmaf(wj, s, -p) + wj * fmaf(res, res, -s);
                        const float n = hi + p, bb = n - hi;
                        lo += (hi - (n - bb)) + (p - bb) + e;
                        hi = n;
                        v[i] = 2.0f * wj * res / (float)ta->B;
                    }
                    put_row(act + qd * kAtom, r, h, v);
                }
                double part = (double)hi + (double)lo;
                const float size = fabsf(hi + lo);
                if (__any_sync(0xffffffffu, !(size <= FLT_MAX) || (size > 0.0f && size < 0x1p-70f))) {
                    part = 0.0;
#pragma unroll 1
                    for (int h = 0; h < 2; h++) {
                        const int c = 64 * qd + 32 * h;
                        if (c >= kOut) break;
                        float v[32];
                        tc::tmem_ld32(tbase + (uint32_t)c, v);
#pragma unroll
                        for (int i = 0; i < 32; i++) {
                            const int j = c + i;
                            if (j >= kOut) continue;
                            const double res = v[i] + __ldg(bias + j) - __ldg(trow + j);
                            part += (double)__ldg(ta->w_out + j) * res * res;
                        }
                    }
                }
                for (int o = 16; o > 0; o >>= 1) part += __shfl_down_sync(0xffffffffu, part, o);
                if (lane == 0 && rank == 0) atomicAdd(ta->loss, part / ta->B);
            }
            publish();
            // backward chain: dz_l = (g W) GELU'(z_l), l = 3 .. 0
            for (int q = kFwd; q < kProducts && ok; q++) {
                const int l = kProducts - 1 - q;
                // (as the biases)
                const float4* gr = reinterpret_cast<const float4*>(ta->s.grad[l]) + row0 * (kHidden / 4) + grad0;
                float4 g4[8];
#pragma unroll
                for (int j = 0; j < 8; j++) g4[j] = gr[j * (32 * kEpiWarps)];
                ok = __all_sync(0xffffffffu, tc::mbar_wait(accum, q & 1, flags));
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                if (!ok) break;
#pragma unroll 1
                for (int h = 0; h < kCols / 32; h++) {
                    if (h > 0) {
#pragma unroll
                        for (int j = 0; j < 8; j++) g4[j] = gr[(8 * h + j) * (32 * kEpiWarps)];
                    }
                    float v[32];
                    tc::tmem_ld32(tbase + (uint32_t)(kCols * qd + 32 * h), v);
#pragma unroll
                    for (int j = 0; j < 8; j++) {
                        v[4 * j] *= g4[j].x;
                        v[4 * j + 1] *= g4[j].y;
                        v[4 * j + 2] *= g4[j].z;
                        v[4 * j + 3] *= g4[j].w;
                    }
                    put_row(atom, r, kPair ? qd & 1 : h, v);
                }
                publish();
            }
        } else if (ok && rank == 0) {
            const bool errs = qa->nets == 1 || blockIdx.y == 1;
            if (qd < 2 && blockIdx.y == 0) {
                // coefficients in data units; the weight ring is free (every MMA has completed)
                float (*tile)[33] = reinterpret_cast<float (*)[33]>(ring + (warp - 2) * 32 * 33 * 4);
#pragma unroll 1
                for (int h = 0; h < 2; h++) {
                    const int c = 64 * qd + 32 * h;
                    float v[32];
                    tc::tmem_ld32(tbase + (uint32_t)c, v);
#pragma unroll
                    for (int i = 0; i < 32; i++) {
                        const float y = v[i] + __ldg(bias + c + i);
                        v[i] = y * __ldg(qa->sd + c + i) + __ldg(qa->mean + c + i);
                    }
                    if (qa->split && row_on) {
                        uint4* hi = reinterpret_cast<uint4*>(qa->split + (row0 + r) * (3 * kCoef) + c);
#pragma unroll
                        for (int j = 0; j < 4; j++) {
                            uint32_t hw[4], lw[4];
#pragma unroll
                            for (int e = 0; e < 4; e++) {
                                const float x0 = v[8 * j + 2 * e], x1 = v[8 * j + 2 * e + 1];
                                hw[e] = pack2(x0, x1);
                                const float2 hf = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&hw[e]));
                                lw[e] = pack2(x0 - hf.x, x1 - hf.y);
                            }
                            const uint4 h4 = make_uint4(hw[0], hw[1], hw[2], hw[3]);
                            hi[j] = h4;
                            hi[kCoef / 8 + j] = h4;
                            hi[2 * kCoef / 8 + j] = make_uint4(lw[0], lw[1], lw[2], lw[3]);
                        }
                    }
                    if (qa->coef) {
                        const int64_t m0 = row0 + 32 * lg;
                        const int rows = (int)(qa->n - m0 < 32 ? qa->n - m0 : 32);
                        tc::store_rows(tile, v, lane, qa->coef + m0 * kCoef, kCoef, 0, rows, c, kCoef);
                    }
                }
            } else if (qd == 2 && errs) {
                float v[32];
                tc::tmem_ld32(tbase + (uint32_t)kCoef, v);
                const float err = exp10f(v[0] + __ldg(bias + kCoef));
                if (row_on) {
                    if (qa->pred_err) qa->pred_err[row0 + r] = err;
                    if (qa->accept) qa->accept[row0 + r] = (in_range && err <= qa->thr_cms) ? 1 : 0;
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if constexpr (kPair) pair_sync();                  // neither leaves while the other may still reach into it
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(256) : "memory");
    }
}

template <bool kPair>
__global__ void __launch_bounds__(kThreads, 1)
k_mlp_train(const __grid_constant__ TrainArgs a, unsigned int* flags) {
    chain<true, kPair>(a.w, &a, nullptr, (int64_t)(blockIdx.x >> (int)kPair) * kRows, flags);
}

__global__ void __launch_bounds__(kThreads, 1)
k_mlp_query(const __grid_constant__ QueryArgs a, unsigned int* flags) {
    chain<false, false>(a.w[blockIdx.y], nullptr, &a, (int64_t)blockIdx.x * kRows, flags);
}

// ---------------------------------------------------------------------------------------
// weight and bias gradients
// ---------------------------------------------------------------------------------------
constexpr int kDwThreads = 192;
constexpr int kDwStage = 3 * 64 * 128;                 // 64 batch rows x (128 + 64) columns
constexpr int kDwStages = 8;
constexpr int kDwSmem = kDwStages * kDwStage + 1024 + 256;
constexpr int kDwTiles = 8 * 4 + 2;                    // layers 1 .. 4: 2 x 4 tiles of 128 x 64; layer 0: 2
constexpr int kBiasGroups = 4 * (kHidden / 8) + kOutPad / 8;     // 8 columns of one layer per warp

// Shared-memory descriptor of an MN-major operand, 128-byte swizzle: a batch row is one 128-byte
// row of 64 columns; blocks of 64 columns lie 8192 bytes apart (leading), groups of 8 batch rows
// 1024 bytes apart (stride).
__device__ __forceinline__ uint64_t sdesc_mn(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFF);
    d |= (uint64_t)(8192 >> 4) << 16;
    d |= (uint64_t)(1024 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

__device__ __forceinline__ void bias_grads(const DwArgs& a, int group) {
    if (group >= kBiasGroups) return;
    const int l = group / (kHidden / 8) < 4 ? group / (kHidden / 8) : 4;
    const int c0 = 8 * (group - l * (kHidden / 8));
    const int ld = l == 4 ? kOutPad : kHidden, rows = l == 4 ? kOut : kHidden;
    const int lane = threadIdx.x & 31;
    // lane sums over every 32nd row, then the lanes: the order the sums have always had
    float s[8];
#pragma unroll
    for (int i = 0; i < 8; i++) s[i] = 0.0f;
    const bf16* g = a.s.gp[l] + (int64_t)lane * ld + c0;
#pragma unroll 8
    for (int b = lane; b < a.B; b += 32, g += 32 * ld) {
        const uint4 v = *reinterpret_cast<const uint4*>(g);
        const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; i++) {
            s[2 * i] += __uint_as_float(u[i] << 16);
            s[2 * i + 1] += __uint_as_float(u[i] & 0xffff0000u);
        }
    }
#pragma unroll
    for (int i = 0; i < 8; i++) {
        for (int o = 16; o > 0; o >>= 1) s[i] += __shfl_down_sync(0xffffffffu, s[i], o);
        if (lane == 0 && c0 + i < rows) a.G[a.offb[l] + c0 + i] = s[i];
    }
}

__global__ void __launch_bounds__(kDwThreads, 1)
k_mlp_dw(const __grid_constant__ DwArgs a, unsigned int* flags) {
    extern __shared__ unsigned char smem_raw[];
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    if (blockIdx.x == 0 && t == 0 && a.advance) {      // read by the kernels before and after this one only
        a.d_step[0] = (a.d_step[0] + 1) % a.steps;
        a.d_step[1] += 1;
    }
    if (blockIdx.x >= kDwTiles) {
        bias_grads(a, (int)(blockIdx.x - kDwTiles) * (kDwThreads / 32) + warp);
        return;
    }
    unsigned char* ring = smem_raw + ((1024u - (tc::smem_u32(smem_raw) & 1023u)) & 1023u);
    uint64_t* full = reinterpret_cast<uint64_t*>(ring + kDwStages * kDwStage);
    uint64_t* empty = full + kDwStages;
    uint64_t* accum = empty + kDwStages;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(accum + 1);
    const int l = blockIdx.x < 32 ? 1 + (int)blockIdx.x / 8 : 0;
    const int q = (int)blockIdx.x - (l == 0 ? 32 : 8 * (l - 1));
    const int m0 = 128 * (l == 0 ? q : q / 4), n0 = 64 * (l == 0 ? 0 : q % 4);
    const int M = l == 4 ? kOut : kHidden, N = l == 0 ? kIn : kHidden;
    const int n_kb = a.B / 64;

    if (t == 0) {
        for (int s = 0; s < kDwStages; s++) { tc::mbar_init(&full[s], 1); tc::mbar_init(&empty[s], 1); }
        tc::mbar_init(accum, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(tc::smem_u32(tmem_slot)), "r"(64) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        if (lane == 0) {
            int armed = 0;
            for (int kb = 0; kb < n_kb; kb++) {
                const int s = kb % kDwStages;
                if (!tc::mbar_wait(&empty[s], ((kb / kDwStages) & 1) ^ 1, flags)) break;
                unsigned char* st = ring + s * kDwStage;
                tc::mbar_expect_tx(&full[s], kDwStage);
                tc::tma_load_2d(st, &a.s.g[l], m0, kb * 64, &full[s]);
                tc::tma_load_2d(st + 8192, &a.s.g[l], m0 + 64, kb * 64, &full[s]);
                tc::tma_load_2d(st + 16384, &a.s.a[l], n0, kb * 64, &full[s]);
                armed = kb + 1;
            }
            for (int kb = armed - 1; kb >= 0 && kb >= armed - kDwStages; kb--)
                tc::mbar_wait(&full[kb % kDwStages], (kb / kDwStages) & 1, flags);
        }
    } else if (warp == 1) {
        if (lane == 0) {
            // both operands MN-major
            constexpr uint32_t idesc = tc::idesc_bf16(64) | (1u << 15) | (1u << 16);
            for (int kb = 0; kb < n_kb; kb++) {
                const int s = kb % kDwStages;
                if (!tc::mbar_wait(&full[s], (kb / kDwStages) & 1, flags)) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t g = tc::smem_u32(ring + s * kDwStage), b = g + 16384;
#pragma unroll
                for (int k = 0; k < 4; k++)            // 16 batch rows a step
                    tc::mma_bf16(tmem, sdesc_mn(g + k * 2048), sdesc_mn(b + k * 2048), idesc, (kb | k) != 0);
                tc::mma_commit(&empty[s]);
            }
            tc::mma_commit(accum);
            tc::mbar_wait(accum, 0, flags);
        }
    } else {
        const int lg = warp & 3;
        const bool done = __all_sync(0xffffffffu, tc::mbar_wait(accum, 0, flags));
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (done) {
            float (*tile)[33] = reinterpret_cast<float (*)[33]>(ring + (warp - 2) * 32 * 33 * 4);
            for (int c = 0; c < 64 && n0 + c < N; c += 32) {
                float v[32];
                tc::tmem_ld32(tmem + ((uint32_t)(32 * lg) << 16) + (uint32_t)c, v);
                tc::store_rows(tile, v, lane, a.G + a.offW[l], N, m0 + 32 * lg, M, n0 + c, N);
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(64) : "memory");
    }
}

// ---------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------
soap_status weight_maps(Weights& w, const bf16* const* W, const bf16* const* WT, const float* const* bias) {
    for (int l = 0; l < kFwd; l++) {
        const int out = l == kFwd - 1 ? kOut : kHidden, in = l == 0 ? kIn : kHidden;
        SOAP_TRY(tc::operand_map(&w.fwd[l], W[l], out, in, in, kHidden / 2));
        w.bias[l] = bias[l];
    }
    for (int q = 0; q < kBwd; q++) {                   // layers 4, 3, 2, 1
        const int l = kFwd - 1 - q, out_pad = l == kFwd - 1 ? kOutPad : kHidden;
        SOAP_TRY(tc::operand_map(&w.bwd[q], WT[l], kHidden, out_pad, out_pad, kHidden / 2));
    }
    return SOAP_OK;
}

soap_status step_maps(Step& s, bf16* const* act, bf16* const* grad, int B) {
    for (int l = 0; l < kFwd; l++) {
        const int na = l == 0 ? kIn : kHidden, ng = l == kFwd - 1 ? kOutPad : kHidden;
        SOAP_TRY(tc::operand_map(&s.a[l], act[l], B, na, na, 64));
        SOAP_TRY(tc::operand_map(&s.g[l], grad[l], B, ng, ng, 64));
        s.gp[l] = grad[l];
    }
    s.x0 = act[0];
    return SOAP_OK;
}

// Pairs while all of them are resident at once (one CTA an SM; a few SMs may have no partner).
static bool pairs_fit(int64_t tiles) {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return false;
    return 2 * tiles <= sms - 8;
}

soap_status train_step(const TrainArgs& a, cudaStream_t st, unsigned int* flags) {
    const int tiles = a.B / kRows;
    const bool pair = pairs_fit(tiles);
    auto* kern = pair ? k_mlp_train<true> : k_mlp_train<false>;
    SOAP_TRY(fit_dynamic_smem(kern, kSmem));
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim = {2, 1, 1};
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(pair ? 2 * tiles : tiles));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kSmem;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = pair ? 1 : 0;
    SOAP_CUDA(cudaLaunchKernelEx(&cfg, kern, a, flags));
    return SOAP_OK;
}

soap_status weight_grads(const DwArgs& a, cudaStream_t st, unsigned int* flags) {
    SOAP_TRY(fit_dynamic_smem(k_mlp_dw, kDwSmem));
    const int bias_blocks = (kBiasGroups + kDwThreads / 32 - 1) / (kDwThreads / 32);
    k_mlp_dw<<<kDwTiles + bias_blocks, kDwThreads, kDwSmem, st>>>(a, flags);
    SOAP_CUDA(cudaGetLastError());
    return SOAP_OK;
}

soap_status query(const QueryArgs& a, cudaStream_t st, unsigned int* flags) {
    SOAP_TRY(fit_dynamic_smem(k_mlp_query, kSmem));
    const int64_t tiles = (a.n + kRows - 1) / kRows;
    if (tiles > INT32_MAX) { set_error("%lld queries in one call", (long long)a.n); return SOAP_ERANGE; }
    k_mlp_query<<<dim3((unsigned)tiles, (unsigned)a.nets), kThreads, kSmem, st>>>(a, flags);
    SOAP_CUDA(cudaGetLastError());
    return SOAP_OK;
}

}  // namespace mlp
}  // namespace soap

// contract_dev.cuh -- device code of the Toeplitz contraction shared by the single-star
// kernels (contract.cu) and the batched persistent kernel (batch.cu).
//
// contract_tile() (the FP64 quiet star, and FP64 contrasts with a row per mu bin; else
// contract_tile_fold64 and contract_tile_fold32) computes one pixel tile of PB phases:
//   out[p][m] = F_q[m] - sum_b Q_p,b * S_q,b [m] + sum_cl C_cl[m] sum_b K_p,cl,b * S_a(cl),b [m]
// (Eqs. 1-4 for the effect `eff`), from a tap table (group starts, per-tap row offsets,
// coefficients [tap][PB]).  One thread owns R pixels m = m0 + threadIdx.x + r*THREADS; acc
// holds F_q - group 0 + folded class terms, tmp one class before its fold.
#pragma once

#include "soap_internal.cuh"

namespace soap {

template <typename T>
struct Rows {
    const T* q;         // quiet rows [n_mu][row_len]
    const T* a[2];      // active rows spot / facula
};

struct ClassTypes {
    int t[SOAP_MAX_CLASSES];
};

struct EffectList {
    int e[3];
};

// PB coefficients of one tap (16-byte vector loads when PB allows; coefficient slabs are
// 256-byte aligned and every job's block is a multiple of PB elements).
template <int PB>
__device__ __forceinline__ void load_coefs(const double* __restrict__ src, double (&cv)[PB]) {
    if constexpr (PB % 2 == 0) {
#pragma unroll
        for (int q = 0; q < PB / 2; q++) {
            const double2 t = __ldg(reinterpret_cast<const double2*>(src) + q);
            cv[2 * q] = t.x; cv[2 * q + 1] = t.y;
        }
    } else {
#pragma unroll
        for (int p = 0; p < PB; p++) cv[p] = __ldg(src + p);
    }
}

// Region classes as the contraction sees them: the type of class cl (which active rows it
// convolves) and its contrast C_cl at pixel m.  TableContrast reads precomputed rows
// [n_class][n_px]; PlanckContrast32 evaluates the Planck ratio of Sect. 4.3.1 in FP32 with the
// same operations as k_contrast32 (so both give the same values, except where load() takes a line).
template <typename T>
struct TableContrast {
    const T* rows;
    int64_t n_px;
    ClassTypes ct;
    __device__ __forceinline__ int type(int cl) const { return ct.t[cl]; }
    __device__ __forceinline__ T at(int cl, int64_t m) const { return rows[(int64_t)cl * n_px + m]; }
    // row k at pixels m .. m + R - 1 (m a multiple of 4; past the last pixel its value)
    template <int R>
    __device__ __forceinline__ void load(int k, int64_t m, int64_t n, T (&c)[R]) const {
        const T* row = rows + (int64_t)k * n_px;
        if ((n_px & 3) == 0 && m + R <= n) {
#pragma unroll
            for (int q = 0; q < R / 4; q++) {
                const float4 v = __ldg(reinterpret_cast<const float4*>(row + m) + q);
                c[4 * q] = v.x; c[4 * q + 1] = v.y; c[4 * q + 2] = v.z; c[4 * q + 3] = v.w;
            }
        } else {
#pragma unroll
            for (int r = 0; r < R; r++) c[r] = row[m + r < n ? m + r : n - 1];
        }
    }
};

struct PlanckContrast32 {
    float aq, fd;            // h c / (lambda_s k T_quiet), grid step Delta
    const int* types;        // [n_class]
    const float* a;          // [n_class]: h c / (lambda_s k T_class)
    int linear;              // load() by a line over every eight pixels
    __device__ __forceinline__ int type(int cl) const { return types[cl]; }
    __device__ __forceinline__ float at(int cl, int64_t m) const {
        // (a pixel index fits 32 bits; a 64-bit integer converts on the FP64 pipe)
        const float inv = expf(-(float)(int)m * fd);       // lambda_s / lambda_m
        return expm1f(aq * inv) / expm1f(a[cl] * inv);
    }
    // At pixels m .. m + R - 1.  Linear between the first and the last of eight pixels where its error,
    // (7 Delta)^2 / 8 |C''| with |C''| <= C x (x + 1) (x the largest Planck exponent; ' by ln lambda),
    // is below 2^-26 C: two evaluations instead of eight.
    template <int R>
    __device__ __forceinline__ void load(int cl, int64_t m, int64_t n, float (&c)[R]) const {
        if (linear) {
            const int64_t m8 = m & ~7ll;
            const float c0 = at(cl, m8), s = (at(cl, m8 + 7) - c0) * (1.0f / 7.0f), r0 = m & 4 ? 4.0f : 0.0f;
#pragma unroll
            for (int r = 0; r < R; r++) c[r] = fmaf(s, r0 + (float)r, c0);
        } else {
#pragma unroll
            for (int r = 0; r < R; r++) c[r] = at(cl, m + r);
        }
    }
};

// bs: per-(group, mu bin) tap starts [G n_mu + 1] (not for the quiet group alone, G = 1): each class is
// folded per bin, acc += C_(cl n_mu + b)[m] . sum_(taps of bin b) (a contrast row per class and bin:
// mu-dependent facula temperatures).
template <int PB, int R, int THREADS, class Con>
__device__ __forceinline__ void contract_tile(int64_t n_px, const Rows<double>& rows, const long long* __restrict__ toff,
                                              const int* __restrict__ gs, int G, const double* __restrict__ cb,
                                              const Con& con, const double* __restrict__ fq, int eff, int64_t tile,
                                              int np, double* __restrict__ out_rows, const int* __restrict__ bs, int n_mu) {
    // Rows are padded past round_up(n_px, 1024) + max tap, so every tap of every pixel of the
    // last tile reads inside its row; only the per-pixel inputs below need a clamped index.
    const int64_t m0 = tile * THREADS * R + threadIdx.x;
    int64_t mcl[R];
#pragma unroll
    for (int r = 0; r < R; r++) {
        const int64_t m = m0 + (int64_t)r * THREADS;
        mcl[r] = m < n_px ? m : n_px - 1;
    }
    // The tap sums accumulate from zero and F_q is added once at the store: every FMA then
    // rounds at the scale of the residual, not of the continuum (about 8x finer in FP32).
    double acc[PB][R];
#pragma unroll
    for (int r = 0; r < R; r++)
#pragma unroll
        for (int p = 0; p < PB; p++) acc[p][r] = 0.0;
    // group 0: subtract (active star) or add (quiet star) the quiet-row convolutions
    {
        const double* base = rows.q + m0;
        const int t1 = gs[1];
#pragma unroll 4
        for (int t = gs[0]; t < t1; t++) {
            const double* row = base + __ldg(toff + t);
            double s[R];
#pragma unroll
            for (int r = 0; r < R; r++) s[r] = __ldg(row + r * THREADS);
            double cv[PB];
            load_coefs<PB>(cb + (int64_t)t * PB, cv);
#pragma unroll
            for (int p = 0; p < PB; p++)
#pragma unroll
                for (int r = 0; r < R; r++) acc[p][r] = fma(cv[p], s[r], acc[p][r]);
        }
    }
    // classes with a contrast row per mu bin: fold each bin's sum separately
    for (int g = 1; g < G; g++) {
        if (gs[g] == gs[g + 1]) continue;
        const int cl = g - 1;
        const double* base = (eff == SOAP_EFFECT_FLUX ? rows.q : rows.a[con.type(cl) == SOAP_FACULA ? 1 : 0]) + m0;
        for (int b = 0; b < n_mu; b++) {
            const int t0 = bs[g * n_mu + b], t1 = bs[g * n_mu + b + 1];
            if (t0 == t1) continue;
            double tmp[PB][R];
#pragma unroll
            for (int p = 0; p < PB; p++)
#pragma unroll
                for (int r = 0; r < R; r++) tmp[p][r] = 0.0;
            for (int t = t0; t < t1; t++) {
                const double* row = base + __ldg(toff + t);
                double s[R];
#pragma unroll
                for (int r = 0; r < R; r++) s[r] = __ldg(row + r * THREADS);
                double cv[PB];
                load_coefs<PB>(cb + (int64_t)t * PB, cv);
#pragma unroll
                for (int p = 0; p < PB; p++)
#pragma unroll
                    for (int r = 0; r < R; r++) tmp[p][r] = fma(cv[p], s[r], tmp[p][r]);
            }
#pragma unroll
            for (int r = 0; r < R; r++) {
                const double cr = eff == SOAP_EFFECT_BCONV ? 1.0 : con.at(cl * n_mu + b, mcl[r]);
#pragma unroll
                for (int p = 0; p < PB; p++) acc[p][r] = fma(cr, tmp[p][r], acc[p][r]);
            }
        }
    }
    // store out_rows[p][m]
#pragma unroll
    for (int p = 0; p < PB; p++) {
        if (p >= np) break;
#pragma unroll
        for (int r = 0; r < R; r++) {
            const int64_t m = m0 + (int64_t)r * THREADS;
            if (m < n_px) out_rows[(int64_t)p * n_px + m] = fq ? fq[mcl[r]] + acc[p][r] : acc[p][r];
        }
    }
}

// Folded form for tap tables without the quiet group (builder mode 2: group g = class g): the
// quiet rows enter each class's operand, X_cl[m - k] = Ca_cl[m] S_a(cl)[m - k] + Cq_cl[m] S_q[m - k]
// with (Ca, Cq) = (C_cl, -1) for the total effect, (0, C_cl - 1) for the flux effect and (1, -1)
// for the convective blueshift effect, so that out[p][m] = F_q[m] + sum_cl sum_taps K X (the
// quiet group's kernel is -sum_cl K_cl): one coefficient vector and one FMA per phase and pixel
// per tap instead of two.  Classes with a contrast row per mu bin keep contract_tile.
// FP64 form, the effect fixed at compile time: X = C S_a - S_q (TOT), S_a - S_q (BCONV),
// (C - 1) S_q (FLUX), one FP64 instruction each (two as fma(a, S_a, b S_q) with the effect's factors
// in registers).  The FP64 pipe is the bound, so the block is small: two phases share the taps of
// either (100 phases x 205,800 pixels, the whole step: 1.48 ms with two phases x four pixels a
// thread, 1.55 with 3 x 2, 1.62 with 4 x 2, 1.8 with 8 x 2; skipping the zero coefficients of larger
// blocks by branches cost more than it saved, 1.60 with 4 x 2).
template <int PB, int R, int THREADS, int EFF, class Con>
__device__ __forceinline__ void contract_tile_fold64(int64_t n_px, const Rows<double>& rows,
                                                     const long long* __restrict__ toff, const int* __restrict__ gs,
                                                     int G, const double* __restrict__ cb, const Con& con,
                                                     const double* __restrict__ fq, int64_t tile, int np,
                                                     double* __restrict__ out_rows) {
    const int64_t m0 = tile * THREADS * R + threadIdx.x;
    int64_t mcl[R];
#pragma unroll
    for (int r = 0; r < R; r++) {
        const int64_t m = m0 + (int64_t)r * THREADS;
        mcl[r] = m < n_px ? m : n_px - 1;
    }
    double acc[PB][R];
#pragma unroll
    for (int p = 0; p < PB; p++)
#pragma unroll
        for (int r = 0; r < R; r++) acc[p][r] = 0.0;
    const double* bq = rows.q + m0;
    for (int g = 0; g < G; g++) {
        const int t0 = gs[g], t1 = gs[g + 1];
        if (t0 == t1) continue;
        const double* ba = rows.a[con.type(g) == SOAP_FACULA ? 1 : 0] + m0;
        double cc[R];                                      // C (TOT) or C - 1 (FLUX)
#pragma unroll
        for (int r = 0; r < R; r++) {
            if constexpr (EFF == SOAP_EFFECT_BCONV) cc[r] = 1.0;
            else if constexpr (EFF == SOAP_EFFECT_FLUX) cc[r] = con.at(g, mcl[r]) - 1.0;
            else cc[r] = con.at(g, mcl[r]);
        }
#pragma unroll 4
        for (int t = t0; t < t1; t++) {
            const long long off = __ldg(toff + t);
            double cv[PB];
            load_coefs<PB>(cb + (int64_t)t * PB, cv);
            double x[R];
#pragma unroll
            for (int r = 0; r < R; r++) {
                const double q = __ldg(bq + off + r * THREADS);
                if constexpr (EFF == SOAP_EFFECT_FLUX) x[r] = cc[r] * q;
                else if constexpr (EFF == SOAP_EFFECT_BCONV) x[r] = __ldg(ba + off + r * THREADS) - q;
                else x[r] = fma(cc[r], __ldg(ba + off + r * THREADS), -q);
            }
#pragma unroll
            for (int p = 0; p < PB; p++) {
#pragma unroll
                for (int r = 0; r < R; r++) acc[p][r] = fma(cv[p], x[r], acc[p][r]);
            }
        }
    }
#pragma unroll
    for (int p = 0; p < PB; p++) {
        if (p >= np) break;
#pragma unroll
        for (int r = 0; r < R; r++) {
            const int64_t m = m0 + (int64_t)r * THREADS;
            if (m < n_px) out_rows[(int64_t)p * n_px + m] = fq ? fq[mcl[r]] + acc[p][r] : acc[p][r];
        }
    }
}

// FP32 form with the effect fixed at compile time: X = C S_a - S_q (TOT), S_a - S_q (BCONV),
// (C - 1) S_q (FLUX, no active row read), from the taps as aligned groups of eight row offsets
// (build_taps_dev).
//
// Tap by tap the loads bound it: two row values a tap and pixel from L1 are 8 + 2 of its cycles a tap
// and 128 pixels, against 5 cycles of FMAs for four phases.  So a thread owns R = 8 consecutive pixels
// and reads the 15 row values that a group's taps need as two 32-byte loads a row (the taps of a class
// and mu bin are about 3.5 consecutive ones, in 1.3 groups of eight); the taps a group lacks are
// skipped by its (uniform) mask.  The phase block's groups and coefficients are staged in shared
// memory, which takes their latency out of the loop, and the registers are held to nine blocks of 64
// threads an SM or more (96 registers, ten blocks): the row loads (60% from L1, the others from L2)
// need the warps more than the next group's values in registers ahead of time.  Taps are added in
// falling order of offset, that is rising tap, with the roundings of the form tap by tap; the
// accumulators of pixel pairs are updated by two-wide FMAs (fma.rn.f32x2: two independent IEEE FMAs).
// A contrast with a row per mu bin (n_sub = n_mu) is a segment of one bin each; it too multiplies the operands
// instead of each bin's sum (61,747 pixels, 37 phases: error against 64 bits 1.0e-6 so, 1.1e-6 by bins).
//
// 100 phases x 205,800 pixels, 3 classes: 73 -> 57 us; 37 phases x 61,747 pixels, a contrast row per
// bin: 66 -> 29 us; batches of 16,834 pixels: 56,060 phases 2.53 -> 1.90 ms, 3,001 single phases
// 382 -> 236 us (both with the contrast by a line, PlanckContrast32: 250 and 85 us of it).
// On the way (the batch of 56,060): 16-byte loads 32 bytes apart 2.77 ms, coefficients from global
// memory 2.41, the next group's values loaded ahead 2.17 at 7 blocks, 8 blocks 2.02, 10 blocks 1.92,
// eight phases a block 2.02, two 2.54, R = 4 2.90, the values shared by neighbouring groups kept 1.97.
__device__ __forceinline__ unsigned long long ct_pack(float lo, float hi) {
    unsigned long long v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(lo), "f"(hi));
    return v;
}
__device__ __forceinline__ void ct_unpack(unsigned long long v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ void ct_fma2(unsigned long long& d, unsigned long long a, unsigned long long b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}

// most aligned groups of a phase block: a run of n taps touches at most ceil((n + 7) / 8)
inline int fold_groups(int n_class, int n_mu, int n_taps) { return n_class * n_mu * ((n_taps + 14) / 8); }

// Shared memory of a block: a chunk of a phase block's groups and coefficients, and two rows of each
// warp's results, skewed so that 16-byte stores of neighbouring threads fall into different banks.
template <int PB, int R, int THREADS>
struct Fold32Smem {
    static constexpr int kChunk = PB <= 4 ? 32 : 128 / PB;
    static constexpr int kRow = 32 * R + (R == 8 ? 32 : 0);
    TapGroup g[kChunk];
    float4 c[kChunk * 8 * PB / 4];
    float4 row[THREADS / 32][2][kRow / 4];
};

// The R + 8 row values from p (a multiple of R values): R = 8 in 32-byte loads, so that a warp's
// addresses are contiguous (16-byte loads 32 bytes apart take twice the L1 cycles).
template <int R>
__device__ __forceinline__ void load_window(const float* __restrict__ p, float (&w)[R + 8]) {
    if constexpr (R == 8) {
#pragma unroll
        for (int k = 0; k < 2; k++)
            asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                : "=f"(w[8 * k]), "=f"(w[8 * k + 1]), "=f"(w[8 * k + 2]), "=f"(w[8 * k + 3]), "=f"(w[8 * k + 4]),
                  "=f"(w[8 * k + 5]), "=f"(w[8 * k + 6]), "=f"(w[8 * k + 7])
                : "l"(p + 8 * k));
    } else {
#pragma unroll
        for (int k = 0; k < R / 4 + 2; k++) {
            const float4 v = __ldg(reinterpret_cast<const float4*>(p) + k);
            w[4 * k] = v.x; w[4 * k + 1] = v.y; w[4 * k + 2] = v.z; w[4 * k + 3] = v.w;
        }
    }
}

template <int PB, int R, int THREADS, int EFF, class Con>
__device__ __forceinline__ void contract_tile_fold32(int64_t n_px, const Rows<float>& rows,
                                                     const TapGroup* __restrict__ grp, int n_grp, int n_sub,
                                                     const float* __restrict__ cb, const Con& con,
                                                     const float* __restrict__ fq, int64_t tile, int np,
                                                     float* __restrict__ out_rows, Fold32Smem<PB, R, THREADS>& sm,
                                                     bool staged) {
    static_assert(R == 4 || R == 8, "consecutive pixels of a thread");
    constexpr int kChunk = Fold32Smem<PB, R, THREADS>::kChunk;
    constexpr bool kActive = EFF != SOAP_EFFECT_FLUX, kCon = EFF != SOAP_EFFECT_BCONV;
    const int64_t m0 = tile * THREADS * R + threadIdx.x * R;
    unsigned long long acc[PB][R / 2];
#pragma unroll
    for (int p = 0; p < PB; p++)
#pragma unroll
        for (int k = 0; k < R / 2; k++) acc[p][k] = 0ull;
    const float* bq = rows.q + m0;
    const float* ba0 = rows.a[0] + m0;
    const float* ba1 = rows.a[1] + m0;
    float cc[R];                                           // C (TOT) or C - 1 (FLUX) of segment `seg`
    int seg = -1;
    for (int c0 = 0; c0 < n_grp; c0 += kChunk) {
        const int nc = min(kChunk, n_grp - c0);
        if (!staged || n_grp > kChunk) {
            __syncthreads();                               // the chunk before is consumed
            for (int i = threadIdx.x; i < nc; i += THREADS) {
                TapGroup d = grp[c0 + i];
                if (con.type(d.tap0 / n_sub) == SOAP_FACULA) d.mask |= 256;
                sm.g[i] = d;
            }
            const float4* src = reinterpret_cast<const float4*>(cb + (int64_t)c0 * (8 * PB));
            for (int i = threadIdx.x; i < nc * (2 * PB); i += THREADS) sm.c[i] = src[i];
            __syncthreads();
        }
#pragma unroll 1
        for (int i = 0; i < nc; i++) {
            const TapGroup d = sm.g[i];
            float Q[R + 8], A[R + 8];
            load_window<R>(bq + d.off4, Q);
            if constexpr (kActive) load_window<R>((d.mask & 256 ? ba1 : ba0) + d.off4, A);
            if constexpr (kCon) {
                if (d.tap0 != seg) {
                    seg = d.tap0;
                    con.template load<R>(seg, m0, n_px, cc);
                    if constexpr (EFF == SOAP_EFFECT_FLUX) {
#pragma unroll
                        for (int r = 0; r < R; r++) cc[r] -= 1.0f;
                    }
                }
            }
            const float* cg = reinterpret_cast<const float*>(sm.c) + i * (8 * PB);
#pragma unroll
            for (int e = 7; e >= 0; e--) {
                if (!((d.mask >> e) & 1)) continue;
                float cv[PB];
                if constexpr (PB % 4 == 0) {
#pragma unroll
                    for (int q = 0; q < PB / 4; q++) {
                        const float4 t = reinterpret_cast<const float4*>(cg + (7 - e) * PB)[q];
                        cv[4 * q] = t.x; cv[4 * q + 1] = t.y; cv[4 * q + 2] = t.z; cv[4 * q + 3] = t.w;
                    }
                } else {
#pragma unroll
                    for (int p = 0; p < PB; p++) cv[p] = cg[(7 - e) * PB + p];
                }
                unsigned long long x2[R / 2];
#pragma unroll
                for (int k = 0; k < R / 2; k++) {
                    float x[2];
#pragma unroll
                    for (int h = 0; h < 2; h++) {
                        const int r = 2 * k + h;
                        if constexpr (EFF == SOAP_EFFECT_FLUX) x[h] = cc[r] * Q[e + r];
                        else if constexpr (EFF == SOAP_EFFECT_BCONV) x[h] = A[e + r] - Q[e + r];
                        else x[h] = fmaf(cc[r], A[e + r], -Q[e + r]);
                    }
                    x2[k] = ct_pack(x[0], x[1]);
                }
#pragma unroll
                for (int p = 0; p < PB; p++) {
                    const unsigned long long c2 = ct_pack(cv[p], cv[p]);
#pragma unroll
                    for (int k = 0; k < R / 2; k++) ct_fma2(acc[p][k], c2, x2[k]);
                }
            }
        }
    }
    // results: rows of a multiple of eight pixels directly, else a warp's 32 R pixels of one phase at
    // a time through its own part of shared memory
    if (R == 8 && (n_px & 7) == 0 && (reinterpret_cast<uintptr_t>(out_rows) & 31) == 0) {
        if (m0 >= n_px) return;
        float base[R];
#pragma unroll
        for (int r = 0; r < R; r++) base[r] = 0.0f;
        if (fq) {
#pragma unroll
            for (int k = 0; k < R / 4; k++) {
                const float4 v = *reinterpret_cast<const float4*>(fq + m0 + 4 * k);
                base[4 * k] = v.x; base[4 * k + 1] = v.y; base[4 * k + 2] = v.z; base[4 * k + 3] = v.w;
            }
        }
#pragma unroll
        for (int p = 0; p < PB; p++) {
            if (p >= np) break;
            float y[R];
#pragma unroll
            for (int k = 0; k < R / 2; k++) ct_unpack(acc[p][k], y[2 * k], y[2 * k + 1]);
            if (fq) {
#pragma unroll
                for (int r = 0; r < R; r++) y[r] = base[r] + y[r];
            }
            if constexpr (R == 8)
                asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(out_rows + (int64_t)p * n_px + m0),
                             "f"(y[0]), "f"(y[1]), "f"(y[2]), "f"(y[3]), "f"(y[4]), "f"(y[5]), "f"(y[6]), "f"(y[7])
                             : "memory");
        }
        return;
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t w0 = tile * THREADS * R + warp * 32 * R + lane;
    float base[R];
#pragma unroll
    for (int k = 0; k < R; k++) base[k] = fq && w0 + 32 * k < n_px ? fq[w0 + 32 * k] : 0.0f;
    __syncwarp();
#pragma unroll
    for (int p = 0; p < PB; p++) {
        if (p >= np) break;
        float* s = reinterpret_cast<float*>(sm.row[warp][p & 1]);
        float* mine = s + lane * R + (R == 8 ? (lane >> 2) * 4 : 0);
#pragma unroll
        for (int k = 0; k < R / 4; k++) {
            float4 v;
            ct_unpack(acc[p][2 * k], v.x, v.y);
            ct_unpack(acc[p][2 * k + 1], v.z, v.w);
            *reinterpret_cast<float4*>(mine + 4 * k) = v;
        }
        __syncwarp();
#pragma unroll
        for (int k = 0; k < R; k++) {
            const int64_t m = w0 + 32 * k;
            const float y = s[32 * k + lane + (R == 8 ? 4 * k : 0)];
            if (m < n_px) out_rows[(int64_t)p * n_px + m] = fq ? base[k] + y : y;
        }
    }
}

// Contrast rows from a device list of temperatures (one row per class and mu bin when facula
// temperatures depend on mu): FP64 rows (and their FP32 copies).
static __global__ void k_contrast_rows(int64_t n_px, double lam_s, double delta, double t_quiet, int n_rows,
                                       const double* __restrict__ temps, double* c64, float* c32) {
    const double hck = kPlanckH * kLightSI / kBoltzmann * 1e10;   // Angstrom Kelvin
    for (int64_t m = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; m < n_px;
         m += (int64_t)gridDim.x * blockDim.x) {
        const double lam = lam_s * exp((double)m * delta);
        const double xq = expm1(hck / (lam * t_quiet));
        for (int k = blockIdx.y; k < n_rows; k += gridDim.y) {
            const double v = xq / expm1(hck / (lam * temps[k]));
            c64[(int64_t)k * n_px + m] = v;
            c32[(int64_t)k * n_px + m] = (float)v;
        }
    }
}

// FP32 rows with the operations of k_contrast32 (a = h c / (lambda_s k T) per row).
static __global__ void k_contrast_rows32(int64_t n_px, float aq, float fd, int n_rows, const float* __restrict__ a,
                                         float* c32) {
    for (int64_t m = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; m < n_px;
         m += (int64_t)gridDim.x * blockDim.x) {
        const float inv = expf(-(float)m * fd);            // lambda_s / lambda_m
        const float xq = expm1f(aq * inv);
        for (int k = blockIdx.y; k < n_rows; k += gridDim.y)
            c32[(int64_t)k * n_px + m] = xq / expm1f(a[k] * inv);
    }
}

// FP32 contrast per class (relative error ~1e-7, inside the mixed path's 2e-6).
struct ClassConsts {
    float a[SOAP_MAX_CLASSES];       // h c / (lambda_s k T_class)
};

static __global__ void k_contrast32(int64_t n_px, float aq, float fd, int n_class, ClassConsts ac, float* c32) {
    for (int64_t m = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; m < n_px;
         m += (int64_t)gridDim.x * blockDim.x) {
        const float inv = expf(-(float)m * fd);            // lambda_s / lambda_m
        const float xq = expm1f(aq * inv);
        for (int cl = 0; cl < n_class; cl++) c32[cl * n_px + m] = xq / expm1f(ac.a[cl] * inv);
    }
}

// ---------------------------------------------------------------------------------------
// regions (Alg. 5): centre, cap and cell box per (phase, region), and the InfoMap owner
// ---------------------------------------------------------------------------------------
struct RegionGeo {
    double P[3];       // unit vector of the cap centre, observer frame
    double cosr;       // cos of the cap's angular radius, sqrt(1 - r^2)
    float Pf[3];
    float cosrf;
    int box[4];        // i0, i1, j0, j1 (empty if i1 < i0)
    int cls;
    int pad;
};

// Region centre at `phase` (observer frame, rotation axis (0, sin i, cos i)): star-frame
// (cos lat sin L, sin lat, cos lat cos L) with L = lon + 360 phase (1 + alpha sin^2 lat), tilted
// by the inclination; written with explicitly rounded FP64 steps.  The cell box is
// conservative: the cap reaches axis angles within +-asin(r) of the centre's.
__device__ __forceinline__ RegionGeo region_geometry(int N, const RegionDev& g, double phase, double incl_deg,
                                                     double alpha) {
    const double d2r = kPi / 180.0;
    const double lat = __dmul_rn(g.lat_deg, d2r);
    double sl, cl;
    sincos(lat, &sl, &cl);
    const double lonp = __dadd_rn(g.lon_deg, __dmul_rn(__dmul_rn(360.0, phase),
                                                       __dadd_rn(1.0, __dmul_rn(__dmul_rn(alpha, sl), sl))));
    const double lon = __dmul_rn(lonp, d2r);
    const double incl = __dmul_rn(incl_deg, d2r);
    double si, ci, sn, cn;
    sincos(incl, &si, &ci);
    sincos(lon, &sn, &cn);
    const double px = __dmul_rn(cl, sn), py = sl, pz = __dmul_rn(cl, cn);
    RegionGeo o;
    o.P[0] = px;
    o.P[1] = __dsub_rn(__dmul_rn(py, si), __dmul_rn(pz, ci));
    o.P[2] = __dadd_rn(__dmul_rn(py, ci), __dmul_rn(pz, si));
    const double r = g.radius;
    o.cosr = __dsqrt_rn(__dsub_rn(1.0, __dmul_rn(r, r)));
    for (int k = 0; k < 3; k++) o.Pf[k] = (float)o.P[k];
    o.cosrf = (float)o.cosr;
    o.cls = g.cls;
    o.pad = 0;
    // The cell box only bounds the cells the exact membership test visits, so it is computed in
    // FP32 (FP64 runs at 1/64 rate here): its error (< 1e-6) is far inside the one-cell margin
    // (2/N), and the far-side cull keeps a 1e-4 rad margin.
    const float pi_f = 3.14159265358979f;
    const float af = asinf(fminf((float)r, 1.0f));
    const float bx = acosf(fmaxf(-1.0f, fminf(1.0f, o.Pf[0])));
    const float by = acosf(fmaxf(-1.0f, fminf(1.0f, o.Pf[1])));
    const float bz = acosf(fmaxf(-1.0f, fminf(1.0f, o.Pf[2])));
    const float xhi = cosf(fmaxf(0.0f, bx - af)), xlo = cosf(fminf(pi_f, bx + af));
    const float yhi = cosf(fmaxf(0.0f, by - af)), ylo = cosf(fminf(pi_f, by + af));
    const float Nf = (float)N;
    int i0 = (int)floorf((xlo * Nf + Nf - 1.0f) * 0.5f) - 1, i1 = (int)ceilf((xhi * Nf + Nf - 1.0f) * 0.5f) + 1;
    int j0 = (int)floorf((ylo * Nf + Nf - 1.0f) * 0.5f) - 1, j1 = (int)ceilf((yhi * Nf + Nf - 1.0f) * 0.5f) + 1;
    i0 = max(i0, 0); j0 = max(j0, 0); i1 = min(i1, N - 1); j1 = min(j1, N - 1);
    if (bz - af > 0.5f * pi_f + 1e-4f) i1 = i0 - 1;     // cap entirely on the far side
    o.box[0] = i0; o.box[1] = i1; o.box[2] = j0; o.box[3] = j1;
    return o;
}

// True when cell (i, j) lies in an earlier region's box (each cell is visited once, from the
// first box that holds it).
__device__ __forceinline__ bool in_earlier_box(const RegionGeo* sg, int r, int i, int j) {
    bool dup = false;
    for (int q = 0; q < r; q++)
        if (i >= sg[q].box[0] && i <= sg[q].box[1] && j >= sg[q].box[2] && j <= sg[q].box[3]) dup = true;
    return dup;
}

// InfoMap owner of a visible cell: a cell (x, y, mu) belongs to a region iff
// (x, y, mu) . P >= sqrt(1 - r^2); the last region in list order that contains it owns it
// (-1: none).  An FP32 test decides cells farther than 2e-6 from the edge (its error is below
// 1e-6); the others are decided by the explicitly rounded FP64 sequence, on the cell centres
// (2 i + 1 - N) / N of the table cellx (IEEE-divided once, as the oracle divides).
// float(v) for |v| < 2^22 without a conversion instruction: the bits 0x4B400000 + v are the float
// 2^23 + 2^22 + v exactly, and one subtraction leaves v.
__device__ __forceinline__ float small_int_to_float(int v) {
    return __int_as_float(0x4B400000 + v) - 12582912.0f;
}

// Box cells in the order t = 0, 1, ... (row-major, width w) for a thread that starts at t0 and
// steps by `step`: the quotient and remainder of the step are taken once, so the walk needs no
// division per cell.
struct BoxWalk {
    int row, col, dq, dr, w;
    __device__ __forceinline__ BoxWalk(int t0, int step, int width) : w(width) {
        row = t0 / width; col = t0 - row * width;
        dq = step / width; dr = step - dq * width;
    }
    __device__ __forceinline__ void next() {
        row += dq; col += dr;
        if (col >= w) { col -= w; row++; }
    }
};

__device__ __forceinline__ int cell_owner(const RegionGeo* sg, int n_regions, int N, float invN, int i, int j,
                                          float muf, const double* __restrict__ cell_mu, int64_t c,
                                          const double* __restrict__ cellx) {
    const float xf = small_int_to_float(2 * i + 1 - N) * invN, yf = small_int_to_float(2 * j + 1 - N) * invN;
    int owner = -1;
    for (int q = 0; q < n_regions; q++) {
        const float df = fmaf(xf, sg[q].Pf[0], fmaf(yf, sg[q].Pf[1], muf * sg[q].Pf[2]));
        bool in;
        if (df > sg[q].cosrf + 2e-6f) in = true;
        else if (df < sg[q].cosrf - 2e-6f) in = false;
        else {
            const double x = cellx[i];
            const double y = cellx[j];
            const double dot = __dadd_rn(__dadd_rn(__dmul_rn(x, sg[q].P[0]), __dmul_rn(y, sg[q].P[1])),
                                         __dmul_rn(cell_mu[c], sg[q].P[2]));
            in = dot >= sg[q].cosr;
        }
        if (in) owner = q;
    }
    return owner;
}

}  // namespace soap

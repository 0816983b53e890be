// convection.cu -- bisector injection (Sect. 4.3, the paper's Convec.model): the line bisector
// of each normalised local spectrum is replaced by a target one (per mu), shifting every point
// by the velocity of its normalised depth.
//
// A point n of depth d = clip(1 - F_n, 0, 1) moves by v = B_row(d) - B_orig(d) (km/s; the
// bisectors are tables over equally spaced depths, linear in between), i.e. to the pixel
// position u_n = n + atanh(v / c) / Delta of the log grid.  The moved points are re-sampled at
// the pixel centres linearly in wavelength, as in Eq. 11: for u_n <= m < u_n+1 the weight is
// expm1((m - u_n) Delta) / expm1((u_n+1 - u_n) Delta); outside the moved range the end values
// repeat.  The moved positions must stay increasing (flagged otherwise).
//
// Linear interpolation is linear, so the two tables merge on the host into one table of
// beta = (B_row - B_orig) / c per row (equal to the two-table form up to rounding), and the
// kernel looks up one value per point.
// k_bisectors: block = (tile of THREADS output pixels, row); the moved positions of the tile and
// a halo covering the largest shift are computed once into shared memory (points off the grid
// hold -inf / +inf), then each thread walks from its own pixel to its bracket: |u_n - n| is below
// halo - 1, so the walk takes about |shift| + 1 steps and never leaves the staged span.  FP64 (the
// local spectra are float64; |v|/c <= 1e-3 keeps atanh and expm1 in their short series).
#include <algorithm>
#include <cmath>
#include <vector>

#include <math_constants.h>

#include "soap_internal.cuh"

namespace soap {

constexpr int kBisThreads = 256;
constexpr int kBisMaxHalo = 64;

__device__ __forceinline__ double table_at(const double* __restrict__ tab, int n_d, double d) {
    const double x = d * (double)(n_d - 1);
    int i = (int)x;                                     // d in [0, 1]: x >= 0
    if (i > n_d - 2) i = n_d - 2;
    const double f = x - (double)i;
    return fma(f, tab[i + 1] - tab[i], tab[i]);
}

// expm1(e) by its series up to e^K (K = 4: |e| <= 1e-4, truncation below 1e-18 of e; K = 6:
// |e| <= 1e-3, below 1e-20 of e), else the library function.
template <int K>
__device__ __forceinline__ double expm1_k(double e) {
    if constexpr (K == 4) {
        return fma(e * e, fma(e, fma(e, 1.0 / 24.0, 1.0 / 6.0), 0.5), e);
    } else if constexpr (K == 6) {
        return expm1_small(e);
    } else {
        return expm1(e);
    }
}

template <int K>
__global__ void __launch_bounds__(kBisThreads)
k_bisectors(const double* __restrict__ in, double* __restrict__ out, int n_px, int n_d,
            const double* __restrict__ beta_tab, double inv_delta, double delta, int halo, unsigned int* flags) {
    __shared__ double su[kBisThreads + 2 * kBisMaxHalo + 2];
    __shared__ double sf[kBisThreads + 2 * kBisMaxHalo + 2];
    const int r = blockIdx.y;
    const double* F = in + (int64_t)r * n_px;
    const double* T = beta_tab + (int64_t)r * n_d;
    const int m0 = blockIdx.x * kBisThreads;
    const int span = kBisThreads + 2 * halo + 1;          // points m0 - halo .. m0 + THREADS + halo
    for (int x = threadIdx.x; x < span; x += kBisThreads) {
        const int n = m0 - halo + x;
        double u = n < 0 ? -CUDART_INF : CUDART_INF, f = 0.0;
        if (n >= 0 && n < n_px) {
            f = F[n];
            const double d = fmin(fmax(1.0 - f, 0.0), 1.0);
            u = (double)n + atanh_small(table_at(T, n_d, d)) * inv_delta;
        }
        su[x] = u;
        sf[x] = f;
    }
    __syncthreads();
    // moved positions must increase (each pair checked once, by the block that owns its left point)
    for (int x = halo + threadIdx.x; x < halo + kBisThreads; x += kBisThreads) {
        const int n = m0 - halo + x;
        if (n >= 0 && n + 1 < n_px && !(su[x + 1] > su[x])) atomicOr(flags, kFlagOrder);
    }
    const int m = m0 + threadIdx.x;
    if (m >= n_px) return;
    // bracket: the largest point k with u_k <= m (-inf at n < 0 ends the walk down by n = m - halo + 1,
    // +inf at n >= n_px ends the walk up by n = m + halo - 1)
    const double mm = (double)m;
    int k = threadIdx.x + halo;
    while (su[k] > mm) k--;
    while (su[k + 1] <= mm) k++;
    double val;
    const int nk = m0 - halo + k;
    if (nk < 0) {
        val = F[0];                                       // before the first moved point
    } else if (nk >= n_px - 1) {
        val = F[n_px - 1];                                // at or past the last moved point
    } else {
        const double w = expm1_k<K>((mm - su[k]) * delta) / expm1_k<K>((su[k + 1] - su[k]) * delta);
        val = fma(w, sf[k + 1] - sf[k], sf[k]);
    }
    out[(int64_t)r * n_px + m] = val;
}

// ---------------------------------------------------------------------------------------
// The usual case, velocities below 1e-5 c and shifts that keep the expm1 arguments below 1e-5.
// ---------------------------------------------------------------------------------------
// The FP64 pipe is the bound (16 cycles a warp instruction and SM), so the kernel spends integer,
// FP32 and shared-memory instructions to save its instructions, 17 a point instead of about 53
// (20 rows x 205,800 pixels: 154 us against 349 with the general kernel):
//  - the depth's table interval comes from the bits of d (n_d - 1), checked against the bits of the
//    interval's ends; base and slope are tabulated in pixels, so the shift is one FMA;
//  - comparisons and clamps are on the bits as integers;
//  - the quotient a / b of the two distances starts from the FP32 reciprocal of b and is refined by
//    its remainder twice (each time squaring the error: 1e-7, 1e-14, below FP64 rounding);
//  - with x = a Delta, y = b Delta, expm1(x) / expm1(y) = (a / b) (1 + (x - y) / 2 + (x - y)(2 x - y) / 12
//    + O(y^3 / 24 < 5e-17)); the second-order term (below 2e-11) and the cubic term of atanh (below
//    4e-11 of the shift) are evaluated in FP32, their errors being below 1e-17.
// Positions are rounded as in the general kernel: u = n + shift.
__device__ __forceinline__ long long order_key(long long b) { return b ^ ((b >> 63) & 0x7fffffffffffffffll); }

// double -> float by its bits (towards zero; values below float's normal range give 0)
__device__ __forceinline__ float bits_to_float(double x) {
    const int hi = __double2hiint(x), lo = __double2loint(x);
    const int mag = (hi & 0x7fffffff) - 0x38000000;
    if (mag < 0x00100000) return 0.0f;
    return __int_as_float((hi & 0x80000000) | (mag << 3) | (int)((unsigned int)lo >> 29));
}
// float -> double by its bits (0 for values below the normal range)
__device__ __forceinline__ double bits_to_double(float x) {
    const int b = __float_as_int(x), mag = b & 0x7fffffff;
    if (mag < 0x00800000) return 0.0;
    return __hiloint2double((b & 0x80000000) | ((mag >> 3) + 0x38000000), b << 29);
}

__global__ void __launch_bounds__(kBisThreads)
k_bisectors_small(const double* __restrict__ in, double* __restrict__ out, int n_rows, int n_px, int n_d,
                  const double2* __restrict__ tab, double half_delta, float d2_12, float d2_3, int halo,
                  unsigned int* flags) {
    __shared__ double su[kBisThreads + 2 * kBisMaxHalo + 2];
    __shared__ double sf[kBisThreads + 2 * kBisMaxHalo + 2];
    const int m0 = blockIdx.x * kBisThreads, m = m0 + (int)threadIdx.x;
    const int span = kBisThreads + 2 * halo + 1;          // points m0 - halo .. m0 + THREADS + halo
    const double depth_scale = (double)(n_d - 1), mm = (double)m;
    const double n_first = (double)(m - halo), n_second = n_first + (double)kBisThreads;
    const long long m_key = __double_as_longlong(mm);
    for (int r = blockIdx.y; r < n_rows; r += gridDim.y) {
        const double* F = in + (int64_t)r * n_px;
        const double2* T = tab + (int64_t)r * n_d;
        __syncthreads();                                  // the row before is consumed
#pragma unroll
        for (int part = 0; part < 2; part++) {
            const int x = threadIdx.x + part * kBisThreads, n = m0 - halo + x;
            if (x >= span) break;
            double u = n < 0 ? -CUDART_INF : CUDART_INF, f = 0.0;
            if (n >= 0 && n < n_px) {
                f = F[n];
                double d = 1.0 - f;
                const long long db = __double_as_longlong(d);
                if (db < 0 || db > 0x7ff0000000000000ll) d = 0.0;          // negative or not a number
                else if (db > 0x3ff0000000000000ll) d = 1.0;
                const double pos = d * depth_scale;
                const long long pb = __double_as_longlong(pos);
                int i = (int)bits_to_float(pos);
                const double lo = bits_to_double((float)i), hi = bits_to_double((float)(i + 1));
                if (pb < __double_as_longlong(lo)) i--;
                else if (pb >= __double_as_longlong(hi)) i++;
                if (i > n_d - 2) i = n_d - 2;
                const double2 t = __ldg(T + i);
                const double s = fma(pos, t.y, t.x);
                const float sf32 = bits_to_float(s);
                u = (part ? n_second : n_first) + (s + bits_to_double(sf32 * sf32 * sf32 * d2_3));
            }
            su[x] = u;
            sf[x] = f;
        }
        __syncthreads();
        // moved positions must increase (each pair checked once, by the block that owns its left point)
        int k = threadIdx.x + halo;
        if (m + 1 < n_px &&
            order_key(__double_as_longlong(su[k + 1])) <= order_key(__double_as_longlong(su[k])))
            atomicOr(flags, kFlagOrder);
        if (m >= n_px) continue;
        // bracket: the largest point k with u_k <= m (negative positions are below any m as integers too)
        while (__double_as_longlong(su[k]) > m_key) k--;
        while (__double_as_longlong(su[k + 1]) <= m_key) k++;
        double val;
        const int nk = m0 - halo + k;
        if (nk < 0) {
            val = F[0];                                   // before the first moved point
        } else if (nk >= n_px - 1) {
            val = F[n_px - 1];                            // at or past the last moved point
        } else {
            const double a = mm - su[k], b = su[k + 1] - su[k], ab = mm - su[k + 1];
            const float af = bits_to_float(a), bf = bits_to_float(b);
            const double r0 = bits_to_double(__frcp_rn(bf));
            double t = a * r0;
            t = fma(fma(-b, t, a), r0, t);
            t = fma(fma(-b, t, a), r0, t);
            const double c = fma(ab, half_delta, bits_to_double((af - bf) * (2.0f * af - bf) * d2_12));
            const double w = fma(t, c, t);
            val = fma(w, sf[k + 1] - sf[k], sf[k]);
        }
        out[(int64_t)r * n_px + m] = val;
    }
}

soap_status inject_bisectors(soap_ctx* c, const double* in, double* out, int n_rows, const double* bis_host,
                             const double* orig_host, int n_d) {
    if (n_rows <= 0) return SOAP_OK;
    double vmax = 0.0;
    for (int64_t i = 0; i < (int64_t)n_rows * n_d; i++) {
        if (!std::isfinite(bis_host[i])) { set_error("bisector table entry %lld not finite", (long long)i); return SOAP_EINVAL; }
        vmax = std::max(vmax, std::fabs(bis_host[i]));
    }
    double omax = 0.0;
    for (int i = 0; i < n_d; i++) {
        if (!std::isfinite(orig_host[i])) { set_error("original bisector entry %d not finite", i); return SOAP_EINVAL; }
        omax = std::max(omax, std::fabs(orig_host[i]));
    }
    const double vbound = vmax + omax;                    // km/s
    if (!(vbound / kCKms <= 1e-3)) { set_error("bisector velocities above 1e-3 c"); return SOAP_ERANGE; }
    const double shift = std::atanh(vbound / kCKms) / c->delta;
    const int halo = (int)std::ceil(shift) + 2;
    if (halo > kBisMaxHalo) {
        set_error("bisector shifts of %.1f pixels exceed %d", shift, kBisMaxHalo - 2);
        return SOAP_ERANGE;
    }
    std::vector<double> beta((size_t)n_rows * n_d);
    for (int r = 0; r < n_rows; r++)
        for (int j = 0; j < n_d; j++)
            beta[(size_t)r * n_d + j] = (bis_host[(size_t)r * n_d + j] - orig_host[j]) / kCKms;
    // largest expm1 argument: (u_n+1 - u_n) Delta <= (1 + 2 shift) Delta
    const double emax = (1.0 + 2.0 * shift) * c->delta;
    // the truncation bounds of the small form, and depth indices exact in FP32
    if (emax <= 1e-5 && vbound / kCKms <= 1e-5 && n_d <= 65536) {
        // per interval of depth: base and slope of the shift (pixels) as a function of d (n_d - 1)
        std::vector<double> lin(2 * (size_t)n_rows * n_d, 0.0);
        for (int r = 0; r < n_rows; r++)
            for (int j = 0; j + 1 < n_d; j++) {
                const double* t = beta.data() + (size_t)r * n_d + j;
                const double slope = (t[1] - t[0]) / c->delta;
                lin[2 * ((size_t)r * n_d + j)] = t[0] / c->delta - j * slope;
                lin[2 * ((size_t)r * n_d + j) + 1] = slope;
            }
        SOAP_TRY(ensure(c->bis_tab, lin.size() * sizeof(double)));
        SOAP_TRY(upload_small(c, c->bis_tab.p, lin.data(), lin.size() * sizeof(double)));
        const unsigned tiles = (unsigned)((c->n_px + kBisThreads - 1) / kBisThreads);
        // the per-thread conversions serve a few rows, while the blocks still fill the GPU
        int dev = 0, sms = 0;
        SOAP_CUDA(cudaGetDevice(&dev));
        SOAP_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        const int per = std::max(1, std::min(4, (int)((int64_t)tiles * n_rows / (sms * 32))));
        const dim3 grid(tiles, (unsigned)std::min(65535, (n_rows + per - 1) / per));
        SOAP_TIMED(c, SOAP_TIMER_BISECTORS,
                   (k_bisectors_small<<<grid, kBisThreads, 0, c->stream>>>(
                       in, out, n_rows, (int)c->n_px, n_d, c->bis_tab.as<double2>(), 0.5 * c->delta,
                       (float)(c->delta * c->delta / 12.0), (float)(c->delta * c->delta / 3.0), halo, c->flags)));
        SOAP_CUDA(cudaGetLastError());
        SOAP_LAUNCHED(c);
        return SOAP_OK;
    }
    SOAP_TRY(ensure(c->bis_tab, beta.size() * sizeof(double)));
    SOAP_TRY(upload_small(c, c->bis_tab.p, beta.data(), beta.size() * sizeof(double)));
    dim3 grid((unsigned)((c->n_px + kBisThreads - 1) / kBisThreads), (unsigned)n_rows);
    auto launch = [&](auto kern) {
        SOAP_TIMED(c, SOAP_TIMER_BISECTORS,
                   (kern<<<grid, kBisThreads, 0, c->stream>>>(in, out, (int)c->n_px, n_d, c->bis_tab.as<double>(),
                                                              1.0 / c->delta, c->delta, halo, c->flags)));
    };
    if (emax <= 1e-4) launch(k_bisectors<4>);
    else if (emax <= 1e-3) launch(k_bisectors<6>);
    else launch(k_bisectors<0>);
    SOAP_CUDA(cudaGetLastError());
    SOAP_LAUNCHED(c);
    return SOAP_OK;
}

}  // namespace soap

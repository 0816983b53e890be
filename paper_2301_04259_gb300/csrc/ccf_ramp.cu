// ccf_ramp.cu -- the line-mask CCF of Sect. 4.1 in FP64 for boxes no wider than a pixel, in one
// multiply-add pair per (line, pixel offset) instead of two, and their overlaps, per (line, velocity).
//
// In the coordinates of ccf.cu, line l at velocity k is the box [U_l + S_k + x, .. + b) with
// x = f_l + g_k in [0, 2) and b <= 1.  As a function of f = f_l alone its overlap with the pixel at
// offset o from U_l is piecewise linear, alpha + beta f, with the pieces
//     x <  1 - b         o = S: b
//     x in [1 - b, 1)    o = S: 1 - x         o = S + 1: x + b - 1
//     x in [1, 2 - b)    o = S + 1: b
//     x in [2 - b, 2)    o = S + 1: 2 - x     o = S + 2: x + b - 2
// Take a unit of lines in the order of their fractions f, and for each offset the running sums
//     A_o = sum w_l F[U_l + o],   B_o = sum w_l f_l F[U_l + o].
// Where f passes the end of a piece of velocity k, the change of its (alpha, beta) times (A_o, B_o)
// is due to CCF(k) (an event); after the last line the last piece times the totals.  The
// velocities are 0.29 pixels apart here, so an offset serves 3.5 of them: 54 offsets x 2
// multiply-adds a line against 177 velocities x 2 pixels and their overlaps.
//
// Block = (some units of lines, 8 spectra); warp = 4 consecutive offsets; lane = (one of them, one
// spectrum).  The unit's pixels are staged as rows of 64 bytes, so a warp reads four neighbouring
// rows, 256 bytes, per line.  A warp's events add into slots of its own, one per velocity it touches,
// which are added up (one or two per velocity) at the end of the block.
//
// What bounds it is the FP64 pipe (one warp instruction per 16 cycles and SM): everything else is
// spent to save its instructions, comparisons of fractions are on their bits as integers, and an
// event that one quarter of a warp executes costs as much as one for all of it, so units are as long
// as shared memory allows.  100 spectra of 205,800 pixels, 12,900 lines, 177 velocities: about
// 0.5 ms, against 1.71 with the windowed kernel (two multiply-adds and ten more FP64 instructions per
// line and velocity for eight spectra).
// Values that the running sums do not give are added line by line by a kernel of their own (k_ramp_direct):
// launched early behind the sums, 0 to 3 us a call where there are none (5 without), 0.35 ms for a NaN in the
// same pixel of all those spectra, 1.3 ms when none of the values can be taken.
//
// Precision (the sums of 1,170 lines against extended precision, root mean square of the relative error over
// velocities): 2.8e-16 for boxes of 0.94 pixels, 5.6e-16 for a quarter of a pixel, 2.0e-15 for a twentieth,
// where the sums that cancel are the larger the narrower the box; overlap by overlap, in chunks of 32
// lines, 1.9e-16, 1.8e-16 and 3.5e-16.
// In FP32, where the instructions around the multiply-adds count, the same form took 125 us for 317
// spectra of 102,901 pixels against 104 of the register-tiled kernel.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "soap_internal.cuh"

namespace soap {

constexpr int kRampMaxLines = 256;      // lines of a unit at most
constexpr int kRampMaxGroups = 32;      // warps of a block
constexpr int kRampRow = 64;            // bytes of a staged pixel

constexpr int kRampSpec = 8;            // spectra per block

struct __align__(16) RampLine { double w, wf; long long key; int U, pad; };     // key: the fraction's bits (it is >= 0)
struct __align__(16) RampEvent { double c1, c2; long long key; unsigned short slot, quarter; int pad; };

static long long ramp_key(double x) {
    long long k;
    memcpy(&k, &x, 8);
    return k;
}

struct RampFinal {              // last pieces of a velocity and its slots (-1: none)
    int slot[2];
    int o[2];                   // offsets from the first one
    double alpha[2], beta[2];
};

// lines [l0 + u L, ..) of unit u in the order of their fractions
__global__ void k_ramp_units(int l0, int l1, int L, const int* __restrict__ U, const double* __restrict__ f64,
                             const double* __restrict__ w64, const int* __restrict__ valid, RampLine* __restrict__ out) {
    __shared__ double sf[kRampMaxLines];
    const int a = l0 + blockIdx.x * L, n = min(L, l1 - a);
    const int i = threadIdx.x;
    if (i < n) sf[i] = f64[a + i];
    __syncthreads();
    if (i >= n) return;
    int rank = 0;
    const double f = sf[i];
    for (int j = 0; j < n; j++) rank += sf[j] < f || (sf[j] == f && j < i);
    const int l = a + i;
    RampLine d;
    d.w = valid[l] ? w64[l] : 0.0;                     // lines whose box leaves the grid: weight zero
    d.wf = d.w * f;
    d.key = __double_as_longlong(f);
    d.U = U[l];
    d.pad = 0;
    out[a - l0 + rank] = d;
}

struct RampArgs {
    const RampLine* lines;
    const RampEvent* events;      // by warp, each list closed by a key above all
    const int* ev_start;                         // [groups + 1]
    const RampFinal* fin;                        // [n_v]
    const int* U;                                // box starts of the lines in mask order, from the first used
    const int* S;                                // [n_v] shifts of the velocities: pixels and fractions
    const double* g;
    const double* spectra;
    double* partial;
    unsigned int* bad;            // [blocks of lines][blocks of spectra]: spectra whose sums are not to be taken
    double box;
    int64_t n_px;
    int n_lines, L, units, per_block, groups, n_events, n_slots, o_min, n_v, n_spec, max_rows;
};

// A running sum also holds the pixels that a velocity's boxes only reach in other pieces, and pixels under
// lines of weight zero; what they add cancels, exactly in exact arithmetic.  An infinity or a NaN does not
// cancel, and a pixel far above the others leaves its rounding behind.  So a block's sums of a spectrum
// are only taken while its largest pixel is finite and within 2^kRampSpread of the geometric mean of its
// pixels that are not zero (by their exponents: whole numbers, a few integer instructions a pixel;
// spectra are within 2^4); k_ramp_direct replaces the others.  At the limit the largest pixel's rounding
// is 2^10 2^-53 of a line's share of the sum, 1e-15 of it with the thousand lines of a block.
constexpr int kRampSpread = 10;

__global__ void __launch_bounds__(32 * kRampMaxGroups, 1)
k_ccf_ramp(const __grid_constant__ RampArgs g, unsigned int* flags) {
    extern __shared__ __align__(16) unsigned char ramp_raw[];
    RampEvent* ev = reinterpret_cast<RampEvent*>(ramp_raw);
    RampLine* lines = reinterpret_cast<RampLine*>(ev + g.n_events);
    double* tot = reinterpret_cast<double*>(lines + g.L);          // [groups][A, B][32]
    double* acc = tot + g.groups * 64;                             // [n_slots][8]
    unsigned char* win = reinterpret_cast<unsigned char*>(acc + g.n_slots * 8);
    // of each spectrum: high word of the largest |pixel| (as ordered; NaN above all), and the number and the
    // exponents' sum of the pixels that are not zero
    __shared__ int s_big[kRampSpec], s_count[kRampSpec];
    __shared__ unsigned long long s_exp[kRampSpec];
    const int t = threadIdx.x, n_thr = blockDim.x, warp = t >> 5, lane = t & 31;
    const int q = lane >> 3, s8 = lane & 7;
    const int s0 = blockIdx.y * kRampSpec, ns = min(kRampSpec, g.n_spec - s0);
    for (int i = t; i < g.n_events; i += n_thr) ev[i] = g.events[i];
    for (int i = t; i < g.groups * 64 + g.n_slots * 8; i += n_thr) tot[i] = 0.0;
    if (t < kRampSpec) s_big[t] = s_count[t] = s_exp[t] = 0;
    int big[2] = {0, 0}, count[2] = {0, 0};            // of the two spectra that this thread stages
    unsigned long long expo[2] = {0, 0};
    const int e0 = warp < g.groups ? g.ev_start[warp] : 0;
    const int u1 = min(g.units, (int)(blockIdx.x + 1) * g.per_block);
    for (int u = blockIdx.x * g.per_block; u < u1; u++) {
        const int l0 = u * g.L, n = min(g.L, g.n_lines - l0);
        const int Umin = g.U[l0];
        const int rows = g.U[l0 + n - 1] - Umin + 4 * g.groups;
        if (rows > g.max_rows) {                       // the host has bounded it
            if (t == 0) atomicOr(flags, kFlagBoxRange);
            continue;
        }
        __syncthreads();                               // the previous unit's rows are consumed
        for (int i = t; i < n; i += n_thr) {
            lines[i] = g.lines[l0 + i];
            lines[i].U -= Umin;
        }
        // four threads per pixel, each a quarter of the row (16 bytes); eight pixels a warp
        const int64_t n_lo = (int64_t)Umin + g.o_min;
        for (int i = t; i < 4 * rows; i += n_thr) {
            const int part = i & 3, x = i >> 2;
            const int64_t pix = n_lo + x;
            const bool on = pix >= 0 && pix < g.n_px;
            const double* src = g.spectra + (int64_t)(s0 + 2 * part) * g.n_px + pix;
            const double v0 = on && 2 * part < ns ? __ldg(src) : 0.0;
            const double v1 = on && 2 * part + 1 < ns ? __ldg(src + g.n_px) : 0.0;
            *reinterpret_cast<double2*>(win + x * kRampRow + 16 * part) = make_double2(v0, v1);
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const int hi = __double2hiint(h ? v1 : v0) & 0x7fffffff;
                big[h] = max(big[h], hi);
                count[h] += hi >= 0x00100000;
                expo[h] += (unsigned int)hi >> 20;
            }
        }
        __syncthreads();
        if (warp < g.groups) {
            const unsigned char* row0 = win + (4 * warp + q) * kRampRow + 8 * s8;
            double A = 0.0, B = 0.0;
            int e = e0;
            RampEvent x = ev[e];
            RampLine next = lines[0];
            double Fn = *reinterpret_cast<const double*>(row0 + next.U * kRampRow);
            auto event = [&]() {
                if (q == x.quarter) {
                    double* a = acc + x.slot * 8 + s8;
                    *a = fma(x.c2, B, fma(x.c1, A, *a));
                }
                __syncwarp();                          // the slot's next event may be another quarter's
                x = ev[++e];
            };
            for (int i = 0; i < n; i++) {
                const RampLine c = next;
                const double F = Fn;
                if (i + 1 < n) {
                    next = lines[i + 1];
                    Fn = *reinterpret_cast<const double*>(row0 + next.U * kRampRow);
                }
                while (x.key <= c.key) event();
                A = fma(c.w, F, A);
                B = fma(c.wf, F, B);
            }
            while (x.quarter < 4) event();             // pieces that end past the last line
            tot[warp * 64 + lane] += A;
            tot[warp * 64 + 32 + lane] += B;
        }
    }
#pragma unroll
    for (int h = 0; h < 2; h++) {
        atomicMax(&s_big[2 * (t & 3) + h], big[h]);
        atomicAdd(&s_count[2 * (t & 3) + h], count[h]);
        atomicAdd(&s_exp[2 * (t & 3) + h], expo[h]);
    }
    __syncthreads();
    // the kernel behind this one may be launched: it waits for this one's end
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // last pieces, slots, one partial row per spectrum
    if (warp == 0) {
        const bool bad = lane < ns && (s_big[lane] >= 0x7ff00000 ||
                                       (int64_t)((s_big[lane] >> 20) - kRampSpread) * s_count[lane] > (int64_t)s_exp[lane]);
        const unsigned int mask = __ballot_sync(0xffffffffu, bad);
        if (lane == 0) g.bad[blockIdx.x * gridDim.y + blockIdx.y] = mask;
    }
    // (lane: velocity lane / 8 of four, spectrum lane mod 8)
    for (int k0 = 4 * warp; k0 < g.n_v; k0 += n_thr / 8) {
        const int k = min(k0 + q, g.n_v - 1);
        const bool on = k0 + q < g.n_v && s8 < ns;
        const RampFinal f = g.fin[k];
        double v = 0.0;
#pragma unroll
        for (int j = 0; j < 2; j++) {
            if (f.slot[j] >= 0) v += acc[f.slot[j] * 8 + s8];
            if (f.o[j] >= 0) {
                const int at = (f.o[j] >> 2) * 64 + 8 * (f.o[j] & 3) + s8;
                v = fma(f.alpha[j], tot[at], v);
                v = fma(f.beta[j], tot[at + 32], v);
            }
        }
        if (on) g.partial[((int64_t)blockIdx.x * g.n_spec + s0 + s8) * g.n_v + k] = v;
    }
}

// The block sums of k_ccf_ramp that are not to be taken, line by line over the pixels that the boxes do
// cover.  Block = (lines and spectra of a block there, 32 velocities); lane = velocity, so that a warp's
// pixels are neighbours; eight warps share the lines.  A box's overlaps are FP64 instructions, which bound
// this: computed once for all spectra, compared on their bits.  Where there is nothing to replace, a block
// only reads its word.
constexpr int kDirectWarps = 8;
__global__ void __launch_bounds__(32 * kDirectWarps)
k_ramp_direct(const __grid_constant__ RampArgs g) {
    __shared__ double part[kDirectWarps][kRampSpec][32];
    // launched early behind k_ccf_ramp, as the reduction behind this one
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int k = 32 * blockIdx.z + lane;
    const unsigned int any = g.bad[blockIdx.x * gridDim.y + blockIdx.y];
    if (any == 0) return;
    const int s0 = blockIdx.y * kRampSpec, kk = min(k, g.n_v - 1), Sk = g.S[kk];
    const double gk = g.g[kk];
    const int u1 = min(g.units, (int)(blockIdx.x + 1) * g.per_block);
    const int l0 = min(g.n_lines, (int)blockIdx.x * g.per_block * g.L), l1 = min(g.n_lines, u1 * g.L);
    double a[kRampSpec];
#pragma unroll
    for (int s = 0; s < kRampSpec; s++) a[s] = 0.0;
    for (int l = l0 + warp; l < l1; l += kDirectWarps) {
        const RampLine c = g.lines[l];
        if ((__double_as_longlong(c.w) << 1) == 0) continue;   // also the lines whose box leaves the grid
        double phi = __longlong_as_double(c.key) + gk;
        const int carry = __double2hiint(phi) >= 0x3ff00000;
        if (carry) phi -= 1.0;
        const double left = 1.0 - phi, rest = phi + g.box - 1.0;
        const double ov = __double_as_longlong(left) < __double_as_longlong(g.box) ? left : g.box;
        const int64_t n = (int64_t)c.U + Sk + carry;
        const bool first = n >= 0 && n < g.n_px;
        const bool second = __double_as_longlong(rest) > 0 && n + 1 >= 0 && n + 1 < g.n_px;
        const double w0 = c.w * ov, w1 = c.w * rest;
        const double* x = g.spectra + (int64_t)s0 * g.n_px + n;
        double X[kRampSpec], Y[kRampSpec];
#pragma unroll
        for (int s = 0; s < kRampSpec; s++) {
            const bool on = (any >> s) & 1;
            X[s] = on && first ? __ldg(x) : 0.0;
            Y[s] = on && second ? __ldg(x + 1) : 0.0;
            x += g.n_px;
        }
#pragma unroll
        for (int s = 0; s < kRampSpec; s++) {
            if (!((any >> s) & 1)) continue;
            a[s] = fma(w0, X[s], a[s]);
            if (second) a[s] = fma(w1, Y[s], a[s]);
        }
    }
#pragma unroll
    for (int s = 0; s < kRampSpec; s++) part[warp][s][lane] = a[s];
    __syncthreads();
    const int s = warp;                                // one spectrum each
    static_assert(kDirectWarps == kRampSpec, "a warp per spectrum");
    double v = 0.0;
#pragma unroll
    for (int w = 0; w < kDirectWarps; w++) v += part[w][s][lane];
    if (((any >> s) & 1) && k < g.n_v) g.partial[((int64_t)blockIdx.x * g.n_spec + s0 + s) * g.n_v + k] = v;
}

// ---------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------
static size_t ramp_fixed_smem(const RampState& r, int L) {
    return (size_t)r.n_events * sizeof(RampEvent) + (size_t)L * sizeof(RampLine) + (size_t)r.groups * 64 * 8 +
           (size_t)r.n_slots * 64;
}

// Events, slots and last pieces of a velocity grid (they do not depend on the lines).
static void ramp_velocities(RampState& r, double v_lo, double v_step, int n_v, double delta, double b,
                            std::vector<RampEvent>& events, std::vector<int>& start, std::vector<RampFinal>& fin) {
    std::vector<int> S((size_t)n_v);
    std::vector<double> gk((size_t)n_v);
    for (int k = 0; k < n_v; k++) {
        const double s = std::atanh((v_lo + (double)k * v_step) / kCKms) / delta;
        const double fl = std::floor(s);
        S[(size_t)k] = (int)fl;
        gk[(size_t)k] = s - fl;
    }
    r.o_min = S[0];
    r.groups = (S[(size_t)n_v - 1] + 2 - r.o_min) / 4 + 1;
    if (r.groups > kRampMaxGroups) return;
    struct E { double th, c1, c2; int o, slot; };
    std::vector<std::vector<E>> by((size_t)r.groups);
    fin.assign((size_t)n_v, RampFinal{});
    int n_slots = 0;
    for (int k = 0; k < n_v; k++) {
        const double g = gk[(size_t)k];
        const int o = S[(size_t)k] - r.o_min;
        // pieces from the one that holds f = 0 on: (end, coefficients at o, o + 1, o + 2)
        struct P { double end, a[3], b[3]; };
        const P pieces[4] = {{1.0 - b - g, {b, 0, 0}, {0, 0, 0}},
                             {1.0 - g, {1.0 - g, g + b - 1.0, 0}, {-1.0, 1.0, 0}},
                             {2.0 - b - g, {0, b, 0}, {0, 0, 0}},
                             {2.0 - g, {0, 2.0 - g, g + b - 2.0}, {0, -1.0, 1.0}}};
        const int first = g < 1.0 - b ? 0 : 1;
        RampFinal f;
        f.slot[0] = n_slots++;
        f.slot[1] = o / 4 != (o + 2) / 4 ? n_slots++ : -1;
        f.o[0] = f.o[1] = -1;
        f.alpha[0] = f.alpha[1] = f.beta[0] = f.beta[1] = 0.0;
        for (int i = first; i < first + 3; i++) {
            const P& p = pieces[i];
            if (i == first + 2) {                      // holds f up to 1
                int n = 0;
                for (int j = 0; j < 3; j++)
                    if (p.a[j] != 0 || p.b[j] != 0) { f.o[n] = o + j; f.alpha[n] = p.a[j]; f.beta[n] = p.b[j]; n++; }
                break;
            }
            const P& z = pieces[i + 1];
            for (int j = 0; j < 3; j++) {
                const double c1 = p.a[j] - z.a[j], c2 = p.b[j] - z.b[j];
                if (c1 == 0 && c2 == 0) continue;
                const int gr = (o + j) / 4;
                by[(size_t)gr].push_back(E{p.end, c1, c2, (o + j) & 3, gr == o / 4 ? f.slot[0] : f.slot[1]});
            }
        }
        fin[(size_t)k] = f;
    }
    r.n_slots = n_slots;
    start.assign(1, 0);
    for (auto& list : by) {
        std::stable_sort(list.begin(), list.end(), [](const E& x, const E& y) { return x.th < y.th; });
        for (const E& e : list) {
            // a piece that ends at or before 0 has ended before the first line: its sums are zero
            events.push_back(RampEvent{e.c1, e.c2, ramp_key(std::max(e.th, 0.0)), (unsigned short)e.slot,
                                       (unsigned short)e.o, 0});
        }
        events.push_back(RampEvent{0, 0, 0x7fffffffffffffffll, 0, 4, 0});
        start.push_back((int)events.size());
    }
    r.n_events = (int)events.size();
}

// Lines per unit and units per block for this mask and number of spectra; p.ramp_L stays 0 where the form
// does not apply.  A unit's rows and tables take one block's whole shared memory: the more lines a unit
// has, the fewer events there are to a line.
soap_status ccf_ramp_plan(soap_ctx* c, CcfState& st, const double* mask_lambda, CcfPlan& p, int sms) {
    RampState& r = st.ramp;
    const double b = 2.0 * p.h;
    if (p.f32 || !(b <= 1.0)) return SOAP_OK;
    const double s_lo = std::atanh(p.v_lo / kCKms) / c->delta;
    const double s_hi = std::atanh((p.v_lo + p.v_step * (p.n_v - 1)) / kCKms) / c->delta;
    if (!((s_hi - s_lo + 4.0) / 4.0 + 1.0 <= kRampMaxGroups) || std::fabs(s_lo) > 1e6 || std::fabs(s_hi) > 1e6) return SOAP_OK;
    const int tiles = (p.n_spec + kRampSpec - 1) / kRampSpec;
    if (tiles > 65535) return SOAP_OK;
    if (!r.ok) {
        // the lines that can be valid (two pixels of margin: the others weigh nothing)
        const double lo = c->lam_s * std::exp((-0.5 - s_lo + p.h - 2.0) * c->delta);
        const double hi = c->lam_s * std::exp(((double)c->n_px - 0.5 - s_hi - p.h + 2.0) * c->delta);
        r.l0 = (int)(std::lower_bound(mask_lambda, mask_lambda + p.n_lines, lo) - mask_lambda);
        r.l1 = (int)(std::upper_bound(mask_lambda, mask_lambda + p.n_lines, hi) - mask_lambda);
        r.plan_tiles = -1;
        std::vector<RampEvent> events;
        std::vector<int> start;
        std::vector<RampFinal> fin;
        ramp_velocities(r, p.v_lo, p.v_step, p.n_v, c->delta, b, events, start, fin);
        if (r.groups > kRampMaxGroups || r.l1 <= r.l0) return SOAP_OK;
        auto al = [](size_t x) { return (x + 255) / 256 * 256; };
        r.o_start = al(events.size() * sizeof(RampEvent));
        r.o_fin = al(r.o_start + start.size() * sizeof(int));
        r.o_lines = al(r.o_fin + fin.size() * sizeof(RampFinal));
        SOAP_TRY(ensure(r.tab, r.o_lines + (size_t)(r.l1 - r.l0) * sizeof(RampLine)));
        char* base = r.tab.as<char>();
        SOAP_TRY(upload_small(c, base, events.data(), events.size() * sizeof(RampEvent)));
        SOAP_TRY(upload_small(c, base + r.o_start, start.data(), start.size() * sizeof(int)));
        SOAP_TRY(upload_small(c, base + r.o_fin, fin.data(), fin.size() * sizeof(RampFinal)));
        r.ok = true;
        r.built_L = 0;
    }
    const int n = r.l1 - r.l0;
    if (r.plan_tiles != tiles) {
        r.plan_tiles = tiles;
        r.L = 0;
        const size_t budget = 224 * 1024;
        // one wave: so many blocks per tile of spectra, the lines spread evenly over them and their units
        const int blocks = std::max(1, sms / tiles), share = (n + blocks - 1) / blocks;
        for (int per = (share + kRampMaxLines - 1) / kRampMaxLines; (share + per - 1) / per >= std::min(n, 16); per++) {
            const int L = (share + per - 1) / per;
            // rows of the unit whose lines spread the most
            double span = 0.0;
            for (int a = 0; a < n; a += L)
                span = std::max(span, std::log(mask_lambda[r.l0 + std::min(n, a + L) - 1] / mask_lambda[r.l0 + a]) / c->delta);
            const double rows = span + 3.0 + 4 * r.groups;
            if (rows * kRampRow + ramp_fixed_smem(r, L) <= budget) {
                r.L = L;
                r.rows = (int)rows;
                r.per_block = per;
                break;
            }
            if (L == 1) break;
        }
    }
    if (!r.L) return SOAP_OK;
    p.ramp_L = r.L;
    p.ramp_rows = r.rows;
    p.ramp_units = (n + r.L - 1) / r.L;
    p.ramp_per_block = r.per_block;
    p.n_chunks = (p.ramp_units + r.per_block - 1) / r.per_block;
    return SOAP_OK;
}

// The unit-ordered line tables (after the line tables they are made from).
soap_status ccf_ramp_build(soap_ctx* c, CcfState& st, const CcfPlan& p) {
    RampState& r = st.ramp;
    if (r.built_L == p.ramp_L) return SOAP_OK;
    k_ramp_units<<<(unsigned)p.ramp_units, kRampMaxLines, 0, c->stream>>>(
        r.l0, r.l1, p.ramp_L, p.U, p.f64, p.w64, p.valid, reinterpret_cast<RampLine*>(r.tab.as<char>() + r.o_lines));
    SOAP_CUDA(cudaGetLastError());
    SOAP_LAUNCHED(c);
    r.built_L = p.ramp_L;
    return SOAP_OK;
}

size_t ccf_ramp_scratch(const CcfPlan& p) {
    return (size_t)p.n_chunks * ((p.n_spec + kRampSpec - 1) / kRampSpec) * sizeof(unsigned int);
}

soap_status ccf_ramp(soap_ctx* c, const CcfState& st, const CcfPlan& p, const double* spectra, double* partial) {
    const RampState& r = st.ramp;
    const char* base = static_cast<const char*>(r.tab.p);
    RampArgs a{};
    a.lines = reinterpret_cast<const RampLine*>(base + r.o_lines);
    a.events = reinterpret_cast<const RampEvent*>(base);
    a.ev_start = reinterpret_cast<const int*>(base + r.o_start);
    a.fin = reinterpret_cast<const RampFinal*>(base + r.o_fin);
    a.U = p.U + r.l0;
    a.S = p.S;
    a.g = p.g64;
    a.bad = p.ramp_bad;
    a.box = 2.0 * p.h;
    a.spectra = spectra;
    a.partial = partial;
    a.n_px = c->n_px;
    a.n_lines = r.l1 - r.l0;
    a.L = p.ramp_L;
    a.units = p.ramp_units;
    a.per_block = p.ramp_per_block;
    a.groups = r.groups;
    a.n_events = r.n_events;
    a.n_slots = r.n_slots;
    a.o_min = r.o_min;
    a.n_v = p.n_v;
    a.n_spec = p.n_spec;
    a.max_rows = p.ramp_rows;
    const size_t smem = ramp_fixed_smem(r, p.ramp_L) + (size_t)p.ramp_rows * kRampRow;
    SOAP_TRY(fit_dynamic_smem(k_ccf_ramp, smem));
    const dim3 grid((unsigned)p.n_chunks, (unsigned)((p.n_spec + kRampSpec - 1) / kRampSpec));
    k_ccf_ramp<<<grid, 32 * std::max(r.groups, 4), smem, c->stream>>>(a, c->flags);
    SOAP_LAUNCHED(c);
    cudaLaunchAttribute attr[1];
    const cudaLaunchConfig_t cfg = pdl_config(dim3(grid.x, grid.y, (unsigned)((p.n_v + 31) / 32)), dim3(32 * kDirectWarps),
                                              c->stream, true, attr);
    SOAP_CUDA(cudaLaunchKernelEx(&cfg, k_ramp_direct, a));     // (the caller counts it)
    return SOAP_OK;
}

}  // namespace soap

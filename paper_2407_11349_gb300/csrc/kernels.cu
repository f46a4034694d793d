// O(N) kernels around the pair sweep: event set-up (validation, tie ranges,
// time blocks), per-call staging of the FP32 event table, per-row finalisation
// (lambda_i, Lambda_i, the gradient of eq. 4) with the global reduction, the rows
// recomputed in FP64, and the cut-posterior location resample (Sec. 2.2).
#include <math_constants.h>

#include "units.cuh"

namespace hk {

// ---------------------------------------------------------------------------
// Set-up: validate the events, per-event source scale, tie ranges, bases.
// ---------------------------------------------------------------------------
__device__ __forceinline__ int64_t lower_bound_d(const double* a, int64_t n, double v) {
    int64_t lo = 0, hi = n;
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (a[mid] < v) lo = mid + 1; else hi = mid;
    }
    return lo;
}

__device__ __forceinline__ int64_t upper_bound_d(const double* a, int64_t n, double v) {
    int64_t lo = 0, hi = n;
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (a[mid] <= v) lo = mid + 1; else hi = mid;
    }
    return lo;
}

__global__ void k_setup(double* t, double* x, double* y, const int32_t* county, int32_t nc,
                        const double* scale_c, int64_t n, int64_t npad, int xy_given, double* is2, float* ces,
                        int32_t* lo, int32_t* hi, double* tb, int* ctr) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < npad;
         e += (int64_t)gridDim.x * blockDim.x) {
        if (e < n) {
            const double te = t[e];
            if (!(te > 0.0) || !isfinite(te) || (e + 1 < n && !(te <= t[e + 1])))
                set_error(ctr, HAWKES_ERR_UNSORTED);
            const int32_t c = county[e];
            double se = 1.0;
            if (c < 0 || c >= nc) set_error(ctr, HAWKES_ERR_ARG);
            else se = scale_c[c];
            if (!(se > 0.0) || !isfinite(se)) set_error(ctr, HAWKES_ERR_ARG);
            is2[e] = 1.0 / (se * se);
            const float ce = static_cast<float>(-2.0 * log2(se));
            ces[e] = ce;
            if (ce > 0.f) atomicMax(ctr + CT_CEMAX, __float_as_int(ce));
            if (xy_given) {
                if (!isfinite(x[e]) || !isfinite(y[e])) set_error(ctr, HAWKES_ERR_ARG);
            } else {
                x[e] = 0.0;
                y[e] = 0.0;
            }
            lo[e] = static_cast<int32_t>(lower_bound_d(t, n, te));
            hi[e] = static_cast<int32_t>(upper_bound_d(t, n, te));
        } else {
            t[e] = t[n - 1];
            x[e] = 0.0;
            y[e] = 0.0;
            is2[e] = 1.0;
            ces[e] = 0.f;
            lo[e] = 0;
            hi[e] = 0;
        }
        if (e % TB == 0) tb[e / TB] = t[e < n ? e : n - 1];
    }
}

// ---------------------------------------------------------------------------
// Per-call constants.
// ---------------------------------------------------------------------------
struct Consts {
    double mu, tx, tt, th, om, h;
    double kx, kt, omt, sr, st, set, seq, cB, cE, itx, itt, iom, ih, beta0;
    bool valid;
};

// One warp forms the constants: the quotients side by side, one per lane, then
// the square roots.  (An FP64 division is a chain of a dozen instructions of
// about 40 cycles; one thread forming them in turn took 6 us.)
__device__ __forceinline__ Consts make_consts(const hawkes_params& P, bool bg_time) {
    Consts k;
    k.mu = P.mu; k.tx = P.tau_x; k.tt = P.tau_t; k.th = P.theta; k.om = P.omega; k.h = P.h;
    k.valid = isfinite(k.mu) && isfinite(k.tx) && isfinite(k.tt) && isfinite(k.th) &&
              isfinite(k.om) && isfinite(k.h) && k.mu >= 0.0 && k.th >= 0.0 && k.tx > 0.0 &&
              k.tt > 0.0 && k.om > 0.0 && k.h > 0.0;
    const int lane = threadIdx.x & 31;
    const double tx2 = k.tx * k.tx, tt2 = k.tt * k.tt, h2 = k.h * k.h;
    double num = 1.0, den = 1.0;
    switch (lane) {
        case 0: num = LOG2E; den = 2.0 * tx2; break;       // a_x
        case 1: num = LOG2E; den = 2.0 * tt2; break;       // a_t
        case 2: num = 2.0 * tx2; den = LOG2E; break;       // 1 / a_x
        case 3: num = 2.0 * tt2; den = LOG2E; break;       // 1 / a_t
        case 4: num = 2.0 * h2; den = LOG2E; break;
        // Space-time background phi2(r; tau_x) phi1(dt; tau_t), or the time-only
        // background phi1(dt; tau_t) / tau_x^2 (eq. 2, tau_x^2 read as the area).
        case 5: den = (bg_time ? 1.0 : TWO_PI) * SQRT_TWO_PI * tx2 * k.tt; break;
        case 6: num = k.om; den = TWO_PI * h2; break;
        case 7: den = k.tx; break;
        case 8: den = k.tt; break;
        case 9: den = k.om; break;
        case 10: den = k.h; break;
        case 11: num = tx2; den = h2; break;
    }
    const double q = num / den, r = sqrt(q);
    auto of = [](double v, int l) { return __shfl_sync(0xffffffffu, v, l); };
    k.kx = of(r, 0);
    k.kt = of(r, 1);
    k.sr = of(q, 2);
    k.st = of(q, 3);
    k.set = of(r, 3);
    k.omt = k.om * LOG2E * k.set;
    k.seq = of(q, 4);
    k.cB = of(q, 5);
    k.cE = of(q, 6);
    k.itx = of(q, 7);
    k.itt = of(q, 8);
    k.iom = of(q, 9);
    k.ih = of(q, 10);
    k.beta0 = of(q, 11);
    return k;
}

// Location draw of event i (cut posterior, Sec. 2.2); below.
__device__ __forceinline__ void draw_location(const EvalDesc& d, int64_t i, uint64_t iteration,
                                              double& x, double& y);

// Zero the accumulators, reset the counters and (FP32 path) stage the event
// table; with `resample`, first draw every event's location (batches: one pass
// over the events instead of two).
// P: device parameters (one per problem), or null to take `pv`.
// model: the HAWKES_MODEL1, HAWKES_BG_TIME and HAWKES_LOGLIK_ONLY bits of the
// call's flags.
// skip: evaluate only tiles whose terms can be nonzero in FP32 (see CC_SKIPDT).
// bctr: the batch's two sweep work cursors to reset, or null.
// Bound by HBM at large n (156 MB at n = 1,000,000); the FP64 constants are
// formed by one warp of each block, because in every warp they would cost more
// than the staging itself.
__global__ void k_prep(const __grid_constant__ EvalDesc one, const EvalDesc* __restrict__ probs,
                       const hawkes_params* __restrict__ P, const __grid_constant__ hawkes_params pv,
                       int model, int stage, int skip, int resample, const uint64_t* d_iteration,
                       int* bctr) {
    const EvalDesc& d = probs ? probs[blockIdx.y] : one;
    const bool model1 = (model & HAWKES_MODEL1) != 0;
    const int64_t n = d.n, npad = d.npad;
    chain_next();
    __shared__ double s_kx, s_kt, s_beta0;
    if (threadIdx.x < 32) {
        const bool bgt = (model & HAWKES_BG_TIME) != 0;
        const Consts k = make_consts(P ? P[blockIdx.y] : pv, bgt);
        s_kx = k.kx;
        s_kt = k.kt;
        s_beta0 = k.beta0;
        if (threadIdx.x == 0 && bctr && blockIdx.x == 0 && blockIdx.y == 0) {
            bctr[CT_WORK] = 0;
            bctr[CT_BAND] = 0;
            bctr[CT_READY] = 0;
            bctr[CT_COUNT + CT_WORK] = 0;
        }
        if (threadIdx.x == 0 && blockIdx.x == 0) {
            double* cc = d.cc;
            int* ctr = d.ctr;
            cc[CC_KX] = k.kx; cc[CC_KT] = k.kt; cc[CC_OMT] = k.omt;
            cc[CC_SR] = k.sr; cc[CC_ST] = k.st; cc[CC_SET] = k.set; cc[CC_SEQ] = k.seq;
            cc[CC_CB] = k.cB; cc[CC_CE] = k.cE;
            cc[CC_MU] = k.mu; cc[CC_TX] = k.tx; cc[CC_TT] = k.tt;
            cc[CC_TH] = k.th; cc[CC_OM] = k.om; cc[CC_H] = k.h;
            cc[CC_TN] = d.t[n - 1];
            // Terms below 2^-126 flush to zero in the FP32 path; rows whose rate is
            // within 1e9 x (n such terms) of that are recomputed in FP64.
            cc[CC_FLAGTHR] = 1e9 * (double)n * 1.1754943508222875e-38 * (k.mu * k.cB + k.th * k.cE);
            // A background term is exactly 0 in FP32 (flush to zero) when its
            // base-2 exponent dt~^2 + r~^2 exceeds 126; an excitation term when
            // omega~ dt~ + beta r~^2 - ce exceeds 126.  With 2 units of margin, a
            // tile whose smallest scaled time gap exceeds both bounds contributes
            // exactly nothing.
            const double cemax = model1 ? 0.0 : static_cast<double>(__int_as_float(ctr[CT_CEMAX]));
            cc[CC_SKIPDTB] = skip ? sqrt(128.0) : 0.0;
            cc[CC_SKIPDT] = skip ? fmax(sqrt(128.0), (cemax + 128.0) / k.omt) : 0.0;
            cc[CC_VALID] = k.valid ? 1.0 : 0.0;
            cc[CC_CEMAX] = cemax;
            cc[CC_BGT] = bgt ? 1.0 : 0.0;
            cc[CC_LLONLY] = (model & HAWKES_LOGLIK_ONLY) ? 1.0 : 0.0;
            for (int q = 0; q < 7; ++q) cc[CC_FTHR + q] = -1.0;
            // coefficients of the row finalisation (see row_lambda)
            const double LB = k.mu * k.cB, LE = k.th * k.cE;
            const double itx = k.itx, itt = k.itt, iom = k.iom, ih = k.ih;
            const double itx3 = itx * itx * itx, itt3 = itt * itt * itt, ih3 = ih * ih * ih;
            cc[CC_LB] = LB;
            cc[CC_LE] = LE;
            cc[CC_A1] = LB * itx3; cc[CC_B1] = 2.0 * LB * itx;
            cc[CC_A2] = LB * itt3; cc[CC_B2] = LB * itt;
            cc[CC_A4] = LE * iom;
            cc[CC_A5] = LE * ih3; cc[CC_B5] = 2.0 * LE * ih;
            cc[CC_ITT] = itt;
            constexpr double F = 1.2e-38;  // 2^-126 = 1.1755e-38, with margin
            cc[CC_F0 + 0] = k.cB * F;
            cc[CC_F0 + 1] = LB * F * ((bgt ? 0.0 : 126.0 * k.sr * itx3) + 2.0 * itx);
            cc[CC_F0 + 2] = LB * F * (126.0 * k.st * itt3 + itt);
            cc[CC_F0 + 3] = k.cE * F;
            cc[CC_F0 + 4] = LE * F * iom;
            cc[CC_F0 + 5] = LE * F * ((cemax + 127.0) * k.seq * ih3 + 2.0 * ih);
            cc[CC_F0 + 6] = LE * F;
            ctr[CT_WORK] = 0;
            ctr[CT_BAND] = 0;
            ctr[CT_READY] = 0;
            ctr[CT_FIX] = 0;
            ctr[CT_DONE] = 0;
            ctr[CT_FDONE] = 0;
            ctr[CT_RDONE] = 0;
            for (int q = 0; q < FIX_DOUBLES; ++q) d.fix7[q] = 0.0;
            if (!k.valid) set_error(ctr, HAWKES_ERR_ARG);
        }
    }
    __syncthreads();
    const double kx = s_kx, kt = s_kt, beta0 = s_beta0;
    const uint64_t iteration = resample ? *d_iteration : 0;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < npad;
         e += (int64_t)gridDim.x * blockDim.x) {
#pragma unroll
        for (int q = 0; q < 6; ++q) d.acc[q * npad + e] = 0.0;
        double xe = 0.0, ye = 0.0;
        if (e < n) {
            if (resample) {
                draw_location(d, e, iteration, xe, ye);
                d.x[e] = xe;
                d.y[e] = ye;
            } else if (stage) {
                xe = d.x[e];
                ye = d.y[e];
            }
        }
        if (!stage) continue;
        float nt, nxh, nxl, nyh, nyl, nb, ce;
        if (e < n) {
            const double tt = (d.t[e] - d.tb[e / TB]) * kt;
            const double xs = xe * kx, ys = ye * kx;
            const float xh = static_cast<float>(xs), yh = static_cast<float>(ys);
            nt = -static_cast<float>(tt);
            nxh = -xh;
            nyh = -yh;
            nxl = -static_cast<float>(xs - static_cast<double>(xh));
            nyl = -static_cast<float>(ys - static_cast<double>(yh));
            nb = -static_cast<float>(model1 ? beta0 : beta0 * d.is2[e]);
            ce = model1 ? 0.f : d.ce[e];
        } else {
            nt = -PAD_T;
            nxh = nyh = nxl = nyl = 0.f;
            nb = 0.f;
            ce = 0.f;
        }
        *rec_q(d.rec, e, 0) = make_float4(nt, nt, nxh, nxh);
        *rec_q(d.rec, e, 1) = make_float4(nxl, nxl, nyh, nyh);
        *rec_q(d.rec, e, 2) = make_float4(nyl, nyl, nb, nb);
        *rec_q(d.rec, e, 3) = make_float4(ce, ce, 0.f, 0.f);
    }
}

// ---------------------------------------------------------------------------
// Row finalisation: lambda_i, clip, Lambda_i and the gradient (FP64).
// S = SB, SBr, SBt, SE, SEt, SEq of row i in natural units (unnormalised).
//
// FP64 arithmetic is the cost (1.7 lanes per clock and SM): the parameters'
// quotients are formed once per call (k_prep), so a row needs one division,
// one logarithm, the exponentials, and the error function only near the ends of
// the time range: erf(a / sqrt 2) rounds to 1 for a > 8.5.
// An exponential whose argument is below -746 is exactly 0.
//
// row_lambda: log lambda_i and the partials of log lambda_i.  With BOUND, b[7] receives a bound on what the FP32 sweep's flushed terms can
// move in the row's outputs.  ex2.approx.ftz returns 0 for every term below
// 2^-126, and a product below 2^-126 in an accumulation flushes too, so each
// FP32 moment sum of row i lacks a nonnegative part that is at most (per
// source, natural units):
//   SB  : F                         SE  : F
//   SBr : F 126 / a_x               SEt : F max(t_i - t_1, 1 / sqrt(a_t))
//   SBt : F 126 / a_t               SEq : F (ce_max + 127) 2 h^2 / log2(e)
// with F = 2^-126 (plus margin for the approximation), summed over the row's
// nb background sources (t_j != t_i) and ne excitation sources (t_j < t_i).
// The r^2 and dt^2 factors follow from 2^-a a <= 126 2^-126 for a >= 126; the
// excitation's from 2^g (ce_max - g) <= 2^-126 (ce_max + 126) for g <= -126.
// The row's outputs are N_k / lambda with N_k linear in the moments, so each
// output moves by at most (|dN_k| + |N_k| dlambda / lambda) / lambda, and the
// log-likelihood by dlambda / lambda.  A clipped row whose true rate could
// reach the clip gets an infinite bound.
// ---------------------------------------------------------------------------
template <bool BOUND>
__device__ __forceinline__ void row_lambda(const double* S, double ti, double t1, double nb, double ne,
                                           const double* __restrict__ cc, double& loglam, double d[6],
                                           double b[7]) {
    const double lam = cc[CC_LB] * S[0] + cc[CC_LE] * S[3];
    for (int q = 0; q < 6; ++q) d[q] = 0.0;
    const double dlam = BOUND ? cc[CC_MU] * cc[CC_F0] * nb + cc[CC_F0 + 6] * ne : 0.0;
    if (lam < CLIP) {
        loglam = log(CLIP);
        if (BOUND)
            for (int q = 0; q < 7; ++q) b[q] = (lam + dlam >= CLIP) ? CUDART_INF : 0.0;
    } else {
        loglam = log(lam);
        const double il = 1.0 / lam;
        d[0] = cc[CC_CB] * S[0] * il;
        d[1] = (cc[CC_A1] * S[1] - cc[CC_B1] * S[0]) * il;
        d[2] = (cc[CC_A2] * S[2] - cc[CC_B2] * S[0]) * il;
        d[3] = cc[CC_CE] * S[3] * il;
        d[4] = (cc[CC_A4] * S[3] - cc[CC_LE] * S[4]) * il;
        d[5] = (cc[CC_A5] * S[5] - cc[CC_B5] * S[3]) * il;
        if (BOUND) {
            const double r = dlam * il, nbl = nb * il, nel = ne * il;
            b[0] = r;
            b[1] = cc[CC_F0] * nbl + fabs(d[0]) * r;
            b[2] = cc[CC_F0 + 1] * nbl + fabs(d[1]) * r;
            b[3] = cc[CC_F0 + 2] * nbl + fabs(d[2]) * r;
            b[4] = cc[CC_F0 + 3] * nel + fabs(d[3]) * r;
            b[5] = (cc[CC_F0 + 4] + cc[CC_F0 + 6] * fmax(ti - t1, cc[CC_SET])) * nel + fabs(d[4]) * r;
            b[6] = cc[CC_F0 + 5] * nel + fabs(d[5]) * r;
        }
    }
    if (cc[CC_LLONLY] != 0.0)  // the sweep formed SB and SE only: no gradient
        for (int q = 0; q < 6; ++q) d[q] = CUDART_NAN;
}

// Lambda_i's three parts (Sec. 2.1) and their derivatives: the Gaussian end
// terms z = Phi(a) - 1/2, w = phi(a) a for a = (t_N - t_i)/tau_t (upper) or
// -t_i/tau_t (lower), and the exponential e^{-omega (t_N - t_i)}.  Only the
// difference of the two z counts, and k_finalize sums each over all rows first:
// without the 1/2 nothing is lost where tau_t is long against the time range and
// the two Phi are nearly equal.
__device__ __forceinline__ void lambda_upper(double ti, const double* __restrict__ cc, double& z, double& w) {
    const double a = (cc[CC_TN] - ti) * cc[CC_ITT], x = 0.5 * a * a;
    z = a > 8.5 ? 0.5 : 0.5 * erf(a * SQRT_HALF);
    w = x > 746.0 ? 0.0 : exp(-x) * 0.3989422804014327 * a;
}
__device__ __forceinline__ void lambda_lower(double ti, const double* __restrict__ cc, double& z, double& w) {
    const double b = -ti * cc[CC_ITT], x = 0.5 * b * b;
    z = b < -8.5 ? -0.5 : 0.5 * erf(b * SQRT_HALF);
    w = x > 746.0 ? 0.0 : exp(-x) * 0.3989422804014327 * b;
}
__device__ __forceinline__ double lambda_exp(double ti, const double* __restrict__ cc, double& gap) {
    gap = cc[CC_TN] - ti;
    const double x = cc[CC_OM] * gap;
    return x > 746.0 ? 0.0 : exp(-x);
}

// A whole row: ell_i, its six partials, log lambda_i, Lambda_i.
__device__ __forceinline__ void row_eval(const double* S, double ti, const double* __restrict__ cc, double out[9]) {
    double d[6], b[7], Pa, Pb, wa, wb, gap;
    row_lambda<false>(S, ti, 0.0, 0.0, 0.0, cc, out[7], d, b);
    lambda_upper(ti, cc, Pa, wa);
    lambda_lower(ti, cc, Pb, wb);
    const double ea = lambda_exp(ti, cc, gap);
    const double mu = cc[CC_MU], th = cc[CC_TH];
    out[8] = mu * (Pa - Pb) + th * (1.0 - ea);
    out[0] = out[7] - out[8];
    out[1] = d[0] - (Pa - Pb);
    out[2] = d[1];
    out[3] = d[2] - mu * (wb - wa) * cc[CC_ITT];
    out[4] = d[3] - (1.0 - ea);
    out[5] = d[4] - th * gap * ea;
    out[6] = d[5];
}

template <int NV>
__device__ __forceinline__ void block_reduce_store(double (&v)[NV], double* dst) {
    __shared__ double red[32][NV];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < NV; ++q)
        for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_down_sync(0xffffffffu, v[q], o);
    if (lane == 0)
        for (int q = 0; q < NV; ++q) red[warp][q] = v[q];
    __syncthreads();
    if (warp == 0) {
        const int nw = blockDim.x >> 5;
        for (int q = 0; q < NV; ++q) {
            double u = lane < nw ? red[lane][q] : 0.0;
            for (int o = 16; o > 0; o >>= 1) u += __shfl_down_sync(0xffffffffu, u, o);
            if (lane == 0) dst[q] = u;
        }
    }
}

// Sums of 16 values over a warp with 16 FP64 additions per lane instead of 80:
// each exchange halves the values a lane still carries.  Lane l returns the
// total of value l >> 1.
__device__ __forceinline__ double warp_sum16(double (&v)[16]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int h = 8, m = 16; h >= 1; h >>= 1, m >>= 1) {
        const bool up = (lane & m) != 0;
#pragma unroll
        for (int k = 0; k < h; ++k) {
            const double keep = up ? v[k + h] : v[k], send = up ? v[k] : v[k + h];
            v[k] = keep + __shfl_xor_sync(0xffffffffu, send, m);
        }
    }
    return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

// The 7 outputs from the totals tot[14] over all rows (outputs, flush bounds)
// and the FP64-recomputed rows' sums; called by one whole block.  The summed
// flush bounds of the FP32 sweep (zero on the FP64 path) decide, per output,
// whether rows must be recomputed by k_flushfix: when an output's bound exceeds
// FLUSH_TAU of its magnitude, every row whose own bound is above FLUSH_TAU
// |output| / nrows is, so the rows left in FP32 can move it by at most
// FLUSH_TAU of its magnitude.
__device__ __forceinline__ void finish_outputs(const double* tot, const volatile double* fix7,
                                               double* cc, int64_t nrows, double* out, int* ctr) {
    const int q = threadIdx.x;
    if (q < 7) {
        const bool valid = cc[CC_VALID] != 0.0, llonly = cc[CC_LLONLY] != 0.0;
        const double r = valid ? tot[q] + fix7[q] : CUDART_NAN;
        out[q] = r;
        const double g = fabs(r), bound = tot[7 + q];
        const bool used = valid && (q == 0 || !llonly);
        if (used && !isfinite(r)) set_error(ctr, HAWKES_ERR_NONFINITE);
        cc[CC_FTHR + q] = (used && bound > FLUSH_TAU * g)
                              ? FLUSH_TAU * g / static_cast<double>(nrows > 0 ? nrows : 1)
                              : -1.0;
    }
}

// Finalise rows [rb, re) (batches: all rows).  With `check` (FP32 sweep), the
// lambda terms of rows whose rate could be moved by FP32 underflow are left
// out and the rows queued for FP64 recomputation, and each block's partials
// also carry the summed flush bounds of its other rows.  The last block to
// finish adds the blocks' partials in a fixed order and writes the 7 outputs
// to out (7 per problem), unless rows were queued: then it keeps the totals for
// k_rows64's last block.
//
// Without per-row outputs (ROWS false) four warps share 32 rows, each forming
// one additive part of their sums: the lambda terms, the two Gaussian end
// terms and the exponential of Lambda.  A warp's chain of FP64 instructions is
// then a third as long, which is what few rows wait for (N = 2,000: 57 us as
// 8 blocks of 256 whole rows, 19.5 in blocks of 64); many rows are bound by
// the FP64 rate either way.
// nparts > 1 (FP64 path): the moment sums are in nparts pieces, parts64[piece][6]
// [rows rounded up to 32] (see k_pairs64).
// err_out (optional): receives the latched error status as a double.
template <bool ROWS>
__global__ void __launch_bounds__(FINAL_THREADS)
    k_finalize(const __grid_constant__ EvalDesc one, const EvalDesc* __restrict__ probs, int64_t rb,
               int64_t re, int check, const double* parts64, int nparts, double* out,
               double* rows9, double* err_out) {
    chain_wait();
    const EvalDesc& d = probs ? probs[blockIdx.y] : one;
    if (probs) {
        rb = 0;
        re = d.n;
        out += 7 * static_cast<int64_t>(blockIdx.y);
    }
    const int64_t n = d.n, npad = d.npad;
    double* cc = d.cc;
    int* ctr = d.ctr;
    double v[16] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
    const bool valid = cc[CC_VALID] != 0.0;
    const double thr = cc[CC_FLAGTHR], LB = cc[CC_LB], LE = cc[CC_LE];
    const double t1 = d.t[0];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int SPAN = ROWS ? FINAL_THREADS : FINAL_THREADS / 4;  // rows per block and step
    const int part = ROWS ? 0 : warp & 3;
    for (int64_t i = rb + static_cast<int64_t>(blockIdx.x) * SPAN + (ROWS ? tid : (warp >> 2) * 32 + lane);
         valid && i < re; i += static_cast<int64_t>(gridDim.x) * SPAN) {
        const double ti = d.t[i], mu = cc[CC_MU], th = cc[CC_TH];
        if (part == 0) {
            double S[6];
            if (nparts > 1) {
                const int64_t stride = (re - rb + 31) / 32 * 32;
                double T[6];  // (two chains, of the first and the last half: less rounding, and side by side)
#pragma unroll
                for (int q = 0; q < 6; ++q) S[q] = parts64[q * stride + i - rb], T[q] = 0.0;
                const int half = nparts / 2;
#pragma unroll 4
                for (int k = 1; k < nparts - half; ++k)
#pragma unroll
                    for (int q = 0; q < 6; ++q) S[q] += parts64[(6 * k + q) * stride + i - rb];
#pragma unroll 4
                for (int k = nparts - half; k < nparts; ++k)
#pragma unroll
                    for (int q = 0; q < 6; ++q) T[q] += parts64[(6 * k + q) * stride + i - rb];
#pragma unroll
                for (int q = 0; q < 6; ++q) S[q] += T[q];
            } else {
#pragma unroll
                for (int q = 0; q < 6; ++q) S[q] = d.acc[q * npad + i];
            }
            const bool queue = check && LB * S[0] + LE * S[3] < thr;
            if (queue) {
                const int k = atomicAdd(ctr + CT_FIX, 1);
                if (kDebug && !(k >= 0 && k < npad))
                    set_error(ctr, HAWKES_ERR_BOUNDS);
                else
                    d.fixlist[k] = static_cast<int>(i);
            } else {
                double loglam, dl[6], bd[7] = {0, 0, 0, 0, 0, 0, 0};
                if (check) {
                    const int64_t l = d.lo[i];
                    row_lambda<true>(S, ti, t1, static_cast<double>(l + (n - d.hi[i])),
                                     static_cast<double>(l), cc, loglam, dl, bd);
                } else {
                    row_lambda<false>(S, ti, t1, 0.0, 0.0, cc, loglam, dl, bd);
                }
                v[0] += loglam;
#pragma unroll
                for (int q = 0; q < 6; ++q) v[1 + q] += dl[q];
                if (check)
#pragma unroll
                    for (int q = 0; q < 7; ++q) v[7 + q] += bd[q];
            }
            if (ROWS && !queue) {  // queued rows are written by k_rows64
                double o[9];
                row_eval(S, ti, cc, o);
                for (int q = 0; q < 9; ++q) rows9[9 * i + q] = o[q];
            }
        }
        if (ROWS || part == 1) {
            double z, w;
            lambda_upper(ti, cc, z, w);
            v[0] -= mu * z;
            v[1] -= z;
            v[3] += mu * w * cc[CC_ITT];
        }
        if (ROWS || part == 2) {
            double z, w;
            lambda_lower(ti, cc, z, w);
            v[0] += mu * z;
            v[1] += z;
            v[3] -= mu * w * cc[CC_ITT];
        }
        if (ROWS || part == 3) {
            double gap;
            const double ea = lambda_exp(ti, cc, gap);
            v[0] -= th * (1.0 - ea);
            v[4] -= 1.0 - ea;
            v[5] -= th * gap * ea;
        }
    }
    chain_next();
    constexpr int NW = FINAL_THREADS / 32;
    __shared__ double red[NW][16];  // per warp; then the totals in red[0]
    __shared__ bool s_last;
    const double w = warp_sum16(v);
    if ((lane & 1) == 0) red[warp][lane >> 1] = w;
    __syncthreads();
    if (tid < 16) {
        double u = red[0][tid];
        for (int k = 1; k < NW; ++k) u += red[k][tid];
        d.partials[PART_STRIDE * blockIdx.x + tid] = u;
        __threadfence();
    }
    __syncthreads();
    if (tid == 0) s_last = atomicAdd(ctr + CT_FDONE, 1) == static_cast<int>(gridDim.x) - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // last block: value tid & 15, every (FINAL_THREADS / 16)-th partial
    const int parts = gridDim.x;
    double u = 0.0;
    for (int b = tid >> 4; b < parts; b += FINAL_THREADS / 16) u += __ldcg(d.partials + PART_STRIDE * b + (tid & 15));
    u += __shfl_xor_sync(0xffffffffu, u, 16);
    if (lane < 16) red[warp][lane] = u;
    __syncthreads();
    if (tid < 16) {
        double s = red[0][tid];
        for (int k = 1; k < NW; ++k) s += red[k][tid];
        red[0][tid] = s;
    }
    __syncthreads();
    const bool queued = valid && *static_cast<volatile int*>(ctr + CT_FIX) > 0;
    if (queued) {
        if (tid < 16) d.fix7[16 + tid] = red[0][tid];
        return;
    }
    finish_outputs(red[0], d.fix7, cc, re - rb, out, ctr);
    __syncthreads();
    if (err_out && tid == 0) *err_out = static_cast<double>(*static_cast<volatile int*>(ctr + CT_ERR));
}

void launch_finalize(cudaStream_t st, dim3 grid, const EvalDesc& one, const EvalDesc* probs, int64_t rb,
                     int64_t re, int check, const double* parts64, int nparts, double* out, double* rows9,
                     double* err_out) {
    launch_chained(rows9 ? k_finalize<true> : k_finalize<false>, grid, FINAL_THREADS, 0, st, one, probs, rb, re, check,
                   parts64, nparts, out, rows9, err_out);
}

// This thread's share (sources j = threadIdx.x + k blockDim.x) of row i's six
// FP64 moment sums, in natural units: the pair terms of eqs. 2-3 written out.
// ix2 = 1/(2 tau_x^2) (0 for the time-only background), it2 = 1/(2 tau_t^2),
// ih2 = 1/(2 h^2).
// The rows that come here are far from all others: nearly every term is an
// exact zero (exp(-v) is 0 in FP64 for v > 745.14), which an FP32 lower bound of v
// above 750 proves without the exponential.  (FP64 arithmetic is 73 times dearer
// than FP32; as in k_pairs64.)  A call with 9,000 sparse events: 234
// -> 143 us.
__device__ __forceinline__ void row_sums64(const EvalDesc& d, int64_t i, bool model1, double ix2,
                                           double it2, double ih2, double om, double v[6]) {
    constexpr float ZERO = 750.f;
    const double ti = d.t[i], xi = d.x[i], yi = d.y[i];
    const int64_t li = d.lo[i], hj = d.hi[i];
    const float ix2f = bound_scale(ix2), it2f = bound_scale(it2), omf = bound_scale(om);
    for (int q = 0; q < 6; ++q) v[q] = 0.0;
    for (int64_t j = threadIdx.x; j < d.n; j += blockDim.x) {
        const double dt = ti - d.t[j], dx = xi - d.x[j], dy = yi - d.y[j];
        const float dtf = bound_diff(dt), dxf = bound_diff(dx), dyf = bound_diff(dy);
        const float r2f = fmaf(dxf, dxf, dyf * dyf);
        // (negated: a NaN is evaluated)
        if ((j < li || j >= hj) && !(fmaf(r2f, ix2f, dtf * dtf * it2f) > ZERO)) {
            const double r2 = dx * dx + dy * dy;
            const double b = exp(-r2 * ix2 - dt * dt * it2);
            v[0] += b;
            v[1] += ix2 != 0.0 ? b * r2 : 0.0;
            v[2] += b * dt * dt;
        }
        if (j < li && !(omf * dtf > ZERO)) {
            const double is2 = model1 ? 1.0 : d.is2[j];
            if (!(fmaf(r2f, bound_scale(ih2 * is2), omf * dtf) > ZERO)) {
                const double r2 = dx * dx + dy * dy;
                const double e = is2 * exp(-om * dt - r2 * ih2 * is2);
                v[3] += e;
                v[4] += e * dt;
                v[5] += e * r2 * is2;
            }
        }
    }
}

// ---------------------------------------------------------------------------
// The rows that k_finalize queued, in FP64: one CTA per row, threads stride over
// all sources; the rows' lambda terms are added into fix7, and the block that
// finishes a problem's last row writes its outputs (see k_finalize).  Returns at
// once when no row is queued.
// nrows: rows of the call (batches: all of the problem).
// A batch's rows are dealt to all blocks whatever problem they belong to, so one
// sparse problem among many has the whole chip (9,000 sparse events among 30
// problems: 23.7 ms with a thirtieth of the blocks for each problem, 1.54 so).
// ---------------------------------------------------------------------------
constexpr int FIX_THREADS = 256;
__global__ void __launch_bounds__(FIX_THREADS)
    k_rows64(const __grid_constant__ EvalDesc one, const EvalDesc* __restrict__ probs, int nprobs, int model,
             int64_t nrows, double* out, double* rows9) {
    chain_wait();
    chain_next();
    if (!probs && (one.cc[CC_VALID] == 0.0 || one.ctr[CT_FIX] == 0)) return;  // (the usual case, without a barrier)
    const bool model1 = (model & HAWKES_MODEL1) != 0;
    __shared__ int queued[FIX_THREADS];  // rows queued by the next problems
    __shared__ double sums[8];
    __shared__ bool s_last;
    const int grid = gridDim.x;
    int turn = blockIdx.x;  // this block's first row of the next problem
    for (int p0 = 0; p0 < nprobs; p0 += FIX_THREADS) {
        int q = 0;
        if (p0 + static_cast<int>(threadIdx.x) < nprobs) {
            const EvalDesc& d = probs ? probs[p0 + threadIdx.x] : one;
            if (d.cc[CC_VALID] != 0.0) q = d.ctr[CT_FIX];
        }
        if (!__syncthreads_or(q)) continue;
        queued[threadIdx.x] = q;
        __syncthreads();
        for (int p = p0; p < min(p0 + FIX_THREADS, nprobs); ++p) {
            const int total = queued[p - p0];
            if (total == 0) continue;
            const EvalDesc& d = probs ? probs[p] : one;
            double* cc = d.cc;
            int* ctr = d.ctr;
            const double tx = cc[CC_TX], tt = cc[CC_TT], om = cc[CC_OM], h = cc[CC_H];
            // Time-only background: no spatial factor in B and no r^2 moment.
            const double ix2 = (model & HAWKES_BG_TIME) ? 0.0 : 1.0 / (2.0 * tx * tx);
            const double it2 = 1.0 / (2.0 * tt * tt), ih2 = 1.0 / (2.0 * h * h);
            int done = 0;
            int64_t k = turn;
            for (; k < total; k += grid, ++done) {
                const int64_t i = d.fixlist[k];
                if (kDebug && !(i >= 0 && i < d.n)) {
                    if (threadIdx.x == 0) set_error(ctr, HAWKES_ERR_BOUNDS);
                    continue;  // uniform over the block: i depends on k only
                }
                double v[6];
                row_sums64(d, i, model1, ix2, it2, ih2, om, v);
                block_reduce_store<6>(v, sums);
                __syncthreads();
                if (threadIdx.x == 0) {
                    // (k_finalize has the row's Lambda terms)
                    double o[9], b[7], loglam, dl[6];
                    row_lambda<false>(sums, d.t[i], 0.0, 0.0, 0.0, cc, loglam, dl, b);
                    atomicAdd(d.fix7, loglam);
                    for (int m = 0; m < 6; ++m) atomicAdd(d.fix7 + 1 + m, dl[m]);
                    if (rows9) {
                        row_eval(sums, d.t[i], cc, o);
                        for (int m = 0; m < 9; ++m) rows9[9 * i + m] = o[m];
                    }
                }
                __syncthreads();
            }
            turn = static_cast<int>(k - total);  // (below the grid: rows go on round the blocks)
            if (done == 0) continue;
            if (threadIdx.x == 0) {
                __threadfence();
                s_last = atomicAdd(ctr + CT_RDONE, done) + done == total;
                __threadfence();
            }
            __syncthreads();
            if (s_last) finish_outputs(d.fix7 + 16, d.fix7, cc, probs ? d.n : nrows, out + (probs ? 7 * static_cast<int64_t>(p) : 0), ctr);
            __syncthreads();
        }
        __syncthreads();
    }
}

// Recompute in FP64 the rows that the flush thresholds (finish_outputs) select
// (a row whose flush bound for some output exceeds that output's threshold;
// rows already recomputed for their low rate are left out), replace their FP32
// values by the FP64 ones in the outputs, and write their per-row values.  Each
// block takes 256-row chunks, a batch's as in k_rows64; the block that finishes a
// problem's last chunk adds the corrections to out.  Returns at once when no
// output needs it (the usual case).
// err_out (optional, one problem): receives the latched error status as a double.
__global__ void __launch_bounds__(FIX_THREADS)
    k_flushfix(const __grid_constant__ EvalDesc one, const EvalDesc* __restrict__ probs, int nprobs, int model,
               int64_t rb, int64_t re, double* out, double* rows9, double* err_out) {
    chain_wait();
    auto wanted = [](const double* cc) {
        bool need = false;
        for (int q = 0; q < 7; ++q) need = need || cc[CC_FTHR + q] >= 0.0;
        return need && cc[CC_VALID] != 0.0;
    };
    if (!probs && !wanted(one.cc)) {  // (the usual case, without a barrier)
        if (err_out && blockIdx.x == 0 && threadIdx.x == 0) *err_out = static_cast<double>(one.ctr[CT_ERR]);
        return;
    }
    const bool model1 = (model & HAWKES_MODEL1) != 0;
    __shared__ bool needed[FIX_THREADS];
    __shared__ int list[FIX_THREADS];
    __shared__ int cnt;
    __shared__ double sums[8];
    __shared__ int last;
    const int grid = gridDim.x;
    int turn = blockIdx.x;  // this block's first chunk of the next problem
    for (int p0 = 0; p0 < nprobs; p0 += FIX_THREADS) {
        bool need = false;
        if (p0 + static_cast<int>(threadIdx.x) < nprobs) need = wanted((probs ? probs[p0 + threadIdx.x] : one).cc);
        if (!__syncthreads_or(need)) continue;
        needed[threadIdx.x] = need;
        __syncthreads();
        for (int p = p0; p < min(p0 + FIX_THREADS, nprobs); ++p) {
            if (!needed[p - p0]) continue;
            const EvalDesc& d = probs ? probs[p] : one;
            const int64_t n = d.n, npad = d.npad;
            const int64_t r0 = probs ? 0 : rb, r1 = probs ? n : re;
            double* o = out + (probs ? 7 * static_cast<int64_t>(p) : 0);
            const double* cc = d.cc;
            int* ctr = d.ctr;
            const double tx = cc[CC_TX], tt = cc[CC_TT], om = cc[CC_OM], h = cc[CC_H];
            const double ix2 = cc[CC_BGT] != 0.0 ? 0.0 : 1.0 / (2.0 * tx * tx);
            const double it2 = 1.0 / (2.0 * tt * tt), ih2 = 1.0 / (2.0 * h * h);
            const double flagthr = cc[CC_FLAGTHR], LB = cc[CC_LB], LE = cc[CC_LE];
            const double t1 = d.t[0];
            double mine[7] = {0, 0, 0, 0, 0, 0, 0};  // thread 0: this block's corrections
            const int64_t chunks = (r1 - r0 + FIX_THREADS - 1) / FIX_THREADS;
            int done = 0;
            int64_t c = turn;
            for (; c < chunks; c += grid, ++done) {
                const int64_t base = r0 + c * FIX_THREADS;
                if (threadIdx.x == 0) cnt = 0;
                __syncthreads();
                const int64_t i = base + threadIdx.x;
                if (i < r1) {
                    double S[6];
                    for (int q = 0; q < 6; ++q) S[q] = d.acc[q * npad + i];
                    if (!(LB * S[0] + LE * S[3] < flagthr)) {
                        double loglam, dl[6], bd[7];
                        const int64_t l = d.lo[i];
                        row_lambda<true>(S, d.t[i], t1, static_cast<double>(l + (n - d.hi[i])),
                                         static_cast<double>(l), cc, loglam, dl, bd);
                        bool f = false;
                        for (int q = 0; q < 7; ++q) f = f || (cc[CC_FTHR + q] >= 0.0 && bd[q] > cc[CC_FTHR + q]);
                        if (f) list[atomicAdd(&cnt, 1)] = threadIdx.x;
                    }
                }
                __syncthreads();
                const int m = cnt;
                for (int k = 0; k < m; ++k) {
                    const int64_t r = base + list[k];
                    double v[6];
                    row_sums64(d, r, model1, ix2, it2, ih2, om, v);
                    block_reduce_store<6>(v, sums);
                    if (threadIdx.x == 0) {
                        double s32[6], d64[6], d32[6], l64, l32, b[7];
                        for (int q = 0; q < 6; ++q) s32[q] = d.acc[q * npad + r];
                        row_lambda<false>(sums, d.t[r], 0.0, 0.0, 0.0, cc, l64, d64, b);
                        row_lambda<false>(s32, d.t[r], 0.0, 0.0, 0.0, cc, l32, d32, b);
                        mine[0] += l64 - l32;
                        for (int q = 0; q < 6; ++q) mine[1 + q] += d64[q] - d32[q];
                        if (rows9) {
                            double o64[9];
                            row_eval(sums, d.t[r], cc, o64);
                            for (int q = 0; q < 9; ++q) rows9[9 * r + q] = o64[q];
                        }
                    }
                    __syncthreads();
                }
            }
            turn = static_cast<int>(c - chunks);
            if (done == 0) continue;
            if (threadIdx.x == 0) {
                for (int q = 0; q < 7; ++q)
                    if (mine[q] != 0.0) atomicAdd(d.fix7 + 8 + q, mine[q]);
                __threadfence();
                last = atomicAdd(ctr + CT_DONE, done) + done == chunks;
            }
            __syncthreads();
            if (last && threadIdx.x == 0) {
                __threadfence();
                const volatile double* fb = d.fix7 + 8;
                const bool llonly = cc[CC_LLONLY] != 0.0;
                bool finite = true;
                for (int q = 0; q < 7; ++q) {
                    const double r = o[q] + fb[q];
                    o[q] = r;
                    if (q == 0 || !llonly) finite = finite && isfinite(r);
                }
                if (!finite) set_error(ctr, HAWKES_ERR_NONFINITE);
                if (err_out) *err_out = static_cast<double>(*static_cast<volatile int*>(ctr + CT_ERR));
            }
            __syncthreads();
        }
        __syncthreads();
    }
}

// Chained and spread over the SMs: where rows are recomputed, their FP64 work
// needs every SM (N = 5,000, sparse: 322 us for the call with the blocks as they
// fall, 252 spread).  nprobs problems (probs), or one (probs null, nprobs 1).
void launch_rows64(cudaStream_t st, int blocks, int sms, const EvalDesc& one, const EvalDesc* probs, int nprobs,
                   int model, int64_t nrows, double* out, double* rows9) {
    launch_chained(k_rows64, blocks, FIX_THREADS, spread_smem(blocks, sms), st, one, probs, nprobs, model, nrows, out,
                   rows9);
}

void launch_flushfix(cudaStream_t st, int blocks, int sms, const EvalDesc& one, const EvalDesc* probs, int nprobs,
                     int model, int64_t rb, int64_t re, double* out, double* rows9, double* err_out) {
    launch_chained(k_flushfix, blocks, FIX_THREADS, spread_smem(blocks, sms), st, one, probs, nprobs, model, rb, re,
                   out, rows9, err_out);
}

cudaError_t rows_setup_attributes() {
    const int most = static_cast<int>(spread_smem(1, 1));
    const cudaError_t e = cudaFuncSetAttribute(k_rows64, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    return e != cudaSuccess ? e
                            : cudaFuncSetAttribute(k_flushfix, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
}

// ---------------------------------------------------------------------------
// Location resample (cut posterior, Sec. 2.2).
// ---------------------------------------------------------------------------
// Triangle areas, evaluated exactly as documented (no fused multiply-add).
__global__ void k_tri_area(const double* __restrict__ xy, int32_t n_tri, double* area, int* ctr) {
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n_tri; k += gridDim.x * blockDim.x) {
        const double* v = xy + 6 * (int64_t)k;
        for (int q = 0; q < 6; ++q)
            if (!isfinite(v[q])) set_error(ctr, HAWKES_ERR_ARG);
        const double cr = __dsub_rn(__dmul_rn(__dsub_rn(v[2], v[0]), __dsub_rn(v[5], v[1])),
                                    __dmul_rn(__dsub_rn(v[4], v[0]), __dsub_rn(v[3], v[1])));
        area[k] = __dmul_rn(0.5, fabs(cr));
    }
}

// Per county: its triangle range and the running area sums (in triangle order).
__global__ void k_tri_county(const int32_t* __restrict__ tri_county, int32_t n_tri,
                             int32_t n_counties, double* cum, int32_t* first, int32_t* last,
                             int* ctr) {
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < n_counties;
         c += gridDim.x * blockDim.x) {
        int lo = 0, hi = n_tri;  // first triangle with county >= c
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (tri_county[mid] < c) lo = mid + 1; else hi = mid;
        }
        int k = lo;
        if (k >= n_tri || tri_county[k] != c) {
            first[c] = -1;
            last[c] = -1;
            set_error(ctr, HAWKES_ERR_ARG);
            continue;
        }
        first[c] = k;
        double run = cum[k];  // cum holds the areas on entry
        for (++k; k < n_tri && tri_county[k] == c; ++k) {
            run = __dadd_rn(run, cum[k]);
            cum[k] = run;
        }
        last[c] = k - 1;
        if (!(run > 0.0)) set_error(ctr, HAWKES_ERR_ARG);
    }
}

__global__ void k_tri_check(const int32_t* __restrict__ tri_county, int32_t n_tri,
                            int32_t n_counties, int* ctr) {
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n_tri; k += gridDim.x * blockDim.x) {
        const int32_t c = tri_county[k];
        if (c < 0 || c >= n_counties || (k > 0 && tri_county[k - 1] > c))
            set_error(ctr, HAWKES_ERR_ARG);
    }
}

// Philox4x64-10 (Salmon et al., SC 2011): ten rounds of two 64x64->128-bit
// multiplies mixing the counter with a Weyl-bumped key.
__device__ __forceinline__ void philox4x64_10(uint64_t c[4], uint64_t k0, uint64_t k1) {
    const uint64_t M0 = 0xD2E7470EE14C6C93ull, M1 = 0xCA5A826395121157ull;
    const uint64_t W0 = 0x9E3779B97F4A7C15ull, W1 = 0xBB67AE8584CAA73Bull;
#pragma unroll
    for (int rd = 0; rd < 10; ++rd) {
        if (rd) {
            k0 += W0;
            k1 += W1;
        }
        const uint64_t hi0 = __umul64hi(M0, c[0]), lo0 = M0 * c[0];
        const uint64_t hi1 = __umul64hi(M1, c[2]), lo1 = M1 * c[2];
        const uint64_t n0 = hi1 ^ c[1] ^ k0, n2 = hi0 ^ c[3] ^ k1;
        c[0] = n0;
        c[1] = lo1;
        c[2] = n2;
        c[3] = lo0;
    }
}

__device__ __forceinline__ double unit53(uint64_t w) {
    return __dmul_rn(static_cast<double>(w >> 11), 1.0 / 9007199254740992.0);
}

__device__ __forceinline__ void draw_location(const EvalDesc& d, int64_t i, uint64_t iteration,
                                              double& x, double& y) {
    const int32_t c = d.county[i];
    uint64_t w[4] = {static_cast<uint64_t>(i), iteration, 0ull, 0ull};
    philox4x64_10(w, d.seed, d.stream);
    const double u0 = unit53(w[0]), u1 = unit53(w[1]), u2 = unit53(w[2]);
    int32_t a = d.cfirst[c], b = d.clast[c];
    const double target = __dmul_rn(u0, d.tri_cum[b]);
    // first k in [a, b] with target < cum[k]; b if there is none
    while (a < b) {
        const int32_t mid = (a + b) >> 1;
        if (target < d.tri_cum[mid]) b = mid; else a = mid + 1;
    }
    const double* v = d.tri_xy + 6 * (int64_t)a;
    const double r1 = __dsqrt_rn(u1);
    const double w0 = __dsub_rn(1.0, r1);
    const double w1 = __dmul_rn(r1, __dsub_rn(1.0, u2));
    const double w2 = __dmul_rn(r1, u2);
    x = __dadd_rn(__dadd_rn(__dmul_rn(w0, v[0]), __dmul_rn(w1, v[2])), __dmul_rn(w2, v[4]));
    y = __dadd_rn(__dadd_rn(__dmul_rn(w0, v[1]), __dmul_rn(w1, v[3])), __dmul_rn(w2, v[5]));
}

__global__ void k_resample(const __grid_constant__ EvalDesc d, uint64_t iteration) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < d.n;
         i += (int64_t)gridDim.x * blockDim.x) {
        double x, y;
        draw_location(d, i, iteration, x, y);
        d.x[i] = x;
        d.y[i] = y;
    }
}

// Self-check of the bounded wait: one thread waits on an mbarrier that nothing
// ever completes; the wait must give up and latch HAWKES_ERR_TIMEOUT.
__global__ void k_wait_selftest(int* ctr) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        fence_barrier_init();
    }
    __syncthreads();
    if (threadIdx.x == 0 && !mbar_wait(&bar, 0)) set_error(ctr, HAWKES_ERR_TIMEOUT);
}

}  // namespace hk

// FP64 pair rows: the six moment sums of eqs. 2-3 for a range of rows, every
// pair term in FP64 (flag HAWKES_F64).
//
// GB300 runs FP64 at 1.7 lanes per clock and SM (measured; FP32 at 124), so the
// number of FP64 instructions is the time, and everything else is free beside
// it.  One warp takes 32 rows, a row per lane, and walks a segment of the
// columns:
//   - For each pair, FP32 arithmetic decides whether a term can be nonzero:
//     exp(-v) is exactly 0 in FP64 for v > 745.14, and a lower bound of v
//     above 750 proves it.  (The FP32 differences are reduced by their rounding,
//     2^-22 of the coordinates' magnitudes; differences too large for FP32 count
//     as 0 and scale factors are rounded down.)  At 1,200 days on 3,000 x 3,000 km
//     that leaves 5% of the background terms and fewer of the excitation.
//   - Each lane queues the columns its row needs, and when a lane's queue is
//     full the warp evaluates all queues, so a warp's FP64 work is that of its
//     pairs and not of every column that some row needs.
//   - exp by a table of 2^(j/512) in two words and a polynomial of degree 4:
//     10 FP64 instructions.
// Every row's terms are added in a fixed order, queue by queue and segment by
// segment, and k_finalize adds the segments in order, so the path is reproducible
// to the last bit.
// Measured at N = 2,000 (100 days, 1,000 x 1,000 km, 82% of the background terms nonzero):
// 424 us as one CTA per row with CUDA's exp over all pairs, 233 here; at
// N = 12,000 over 1,200 days 13.1 ms and 0.92 ms.
#include <algorithm>

#include "units.cuh"
#include "exp_table.cuh"

namespace hk {

// exp(x) for x <= 0 (Tang, "Table-driven implementation of the exponential
// function in IEEE floating-point arithmetic", 1989): x = k ln2 / 512 + r,
// |r| <= ln2 / 1024, exp(x) = 2^(k div 512) 2^((k mod 512) / 512) e^r.  The table
// holds 2^(j/512) as a rounded double and the rest; the polynomial's truncation
// is below 2e-18, so the error is the final rounding's half ulp and little more.

__device__ __forceinline__ double exp_neg(double x, const double2* __restrict__ tab) {
    const int xh = __double2hiint(x) & 0x7fffffff;
    if (xh > 0x40877000) return xh > 0x7ff00000 ? x : 0.0;  // below -750 (or NaN)
    const double t = fma(x, 0x1.71547652b82fep+9, 6755399441055744.0);  // 512 / ln 2; rounds to an integer
    const int k = __double2loint(t);
    const double kd = t - 6755399441055744.0;
    double r = fma(kd, -0x1.62e42fefa39efp-10, x);  // ln 2 / 512
    r = fma(kd, -0x1.abc9e3b39803fp-65, r);
    double q = fma(r, 1.0 / 24.0, 1.0 / 6.0);
    q = fma(r, q, 0.5);
    const double p = fma(r * r, q, r);
    const double2 T = tab[k & (EXP_N - 1)];
    double y = T.x + fma(T.x, p, T.y);
    const int m = k >> 9;
    if (m > -1022) return __hiloint2double(__double2hiint(y) + (m << 20), __double2loint(y));
    y = __hiloint2double(__double2hiint(y) + ((m + 512) << 20), __double2loint(y));  // subnormal result
    return y * 0x1p-512;
}

constexpr int R64_WARPS = 8;  // most warps per CTA (one CTA per SM)
constexpr int R64_QB = 16, R64_QE = 8;  // queued columns per lane
constexpr int R64_FOLD = 16;            // queues per second-level sum
constexpr float R64_ZERO = 750.f;

struct R64Warp {
    float4 col[32];  // x, y, t (FP32, from the reference point), 1 / (2 h^2 s_j^2)
    int qb[R64_QB][32], qe[R64_QE][32];
};

// |a - b| less the rounding of both, at least 0.
__device__ __forceinline__ float low_diff(float a, float b) {
    return fmaxf(0.f, fabsf(a - b) - 2.384185791015625e-07f * (fabsf(a) + fabsf(b)));
}

// FP32 form of a difference; one whose square could overflow becomes NaN, which
// low_diff turns into 0.
__device__ __forceinline__ float bound_coord(double a) {
    return fabs(a) < 1e18 ? static_cast<float>(a) : __int_as_float(0x7fc00000);
}
// Items: (group of 32 rows from row_begin, segment of the columns).  Sums go to
// out[(segment * 6 + moment) * stride + row - origin].
template <bool BGT>
__global__ void __launch_bounds__(32 * R64_WARPS, 1)
    k_pairs64(const __grid_constant__ EvalDesc d, int model1, int64_t row_begin, int64_t row_end, int groups,
              int segments, double* __restrict__ out, int64_t stride, int64_t origin) {
    extern __shared__ __align__(16) unsigned char smem[];
    double2* tab = reinterpret_cast<double2*>(smem);
    R64Warp* warps = reinterpret_cast<R64Warp*>(smem + EXP_N * sizeof(double2));
    const double* cc = d.cc;
    chain_wait();
    if (cc[CC_VALID] == 0.0) return;
    for (int k = threadIdx.x; k < EXP_N; k += blockDim.x) tab[k] = kExpTable[k];
    __syncthreads();
    const int lane = threadIdx.x & 31;
    R64Warp& w = warps[threadIdx.x >> 5];
    constexpr unsigned ALL = 0xffffffffu;
    const double tx = cc[CC_TX], tt = cc[CC_TT], om = cc[CC_OM], h = cc[CC_H];
    // Time-only background: no spatial factor in B and no r^2 moment.
    const double ix2 = BGT ? 0.0 : 1.0 / (2.0 * tx * tx), it2 = 1.0 / (2.0 * tt * tt), ih2 = 1.0 / (2.0 * h * h);
    const float ix2f = bound_scale(ix2), it2f = bound_scale(it2), omf = bound_scale(om);
    const int64_t n = d.n;
    const int64_t seg = ((n + segments - 1) / segments + 31) / 32 * 32;
    for (;;) {
        int item = 0;
        if (lane == 0) item = atomicAdd(d.ctr + CT_WORK, 1);
        item = __shfl_sync(ALL, item, 0);
        if (item >= groups * segments) {
            chain_next();
            return;
        }
        const int g = item / segments, sg = item % segments;
        const int64_t i = row_begin + 32 * static_cast<int64_t>(g) + lane;
        const bool live = i < row_end;
        const int64_t ir = live ? i : row_end - 1;
        const double ti = d.t[ir], xi = d.x[ir], yi = d.y[ir];
        const int lo = live ? d.lo[ir] : 0, hi = live ? d.hi[ir] : 0x7fffffff;  // (no column: no term)
        // reference point of the FP32 tests: the group's first row
        const double x0 = __shfl_sync(ALL, xi, 0), y0 = __shfl_sync(ALL, yi, 0), t0 = __shfl_sync(ALL, ti, 0);
        const float xf = bound_coord(xi - x0), yf = bound_coord(yi - y0), tf = bound_coord(ti - t0);
        // The row's sums, in two levels so that no chain of additions grows with the
        // events: R64_FOLD queues (v), and those (total).
        double v[6] = {0, 0, 0, 0, 0, 0}, total[6] = {0, 0, 0, 0, 0, 0};
        int queues = 0;      // evaluated since the last fold
        int nb = 0, ne = 0;  // queued columns of this lane's row
        auto add = [&]() {
            if (++queues < R64_FOLD) return;
            queues = 0;
            for (int q = 0; q < 6; ++q) {
                total[q] += v[q];
                v[q] = 0.0;
            }
        };

        auto term_b = [&](int j) {
            const double dt = ti - d.t[j];
            const double dt2 = dt * dt;
            if (BGT) {
                const double b = exp_neg(-dt2 * it2, tab);
                v[0] += b;
                v[2] = fma(b, dt2, v[2]);
            } else {
                const double dx = xi - d.x[j], dy = yi - d.y[j];
                const double r2 = fma(dy, dy, dx * dx);
                const double b = exp_neg(-fma(r2, ix2, dt2 * it2), tab);
                v[0] += b;
                v[1] = fma(b, r2, v[1]);
                v[2] = fma(b, dt2, v[2]);
            }
        };
        auto eval_b = [&]() {
            if (__all_sync(ALL, nb == R64_QB)) {  // every lane: independent chains side by side
#pragma unroll 4
                for (int k = 0; k < R64_QB; ++k) term_b(w.qb[k][lane]);
            } else {
                const int m = __reduce_max_sync(ALL, nb);
                for (int k = 0; k < m; ++k)
                    if (k < nb) term_b(w.qb[k][lane]);
            }
            add();
            nb = 0;
            __syncwarp();
        };
        auto eval_e = [&]() {
            const int m = __reduce_max_sync(ALL, ne);
            for (int k = 0; k < m; ++k)
                if (k < ne) {
                    const int j = w.qe[k][lane];
                    const double is2 = model1 ? 1.0 : d.is2[j];
                    const double dt = ti - d.t[j], dx = xi - d.x[j], dy = yi - d.y[j];
                    const double q = fma(dy, dy, dx * dx) * is2;
                    const double e = is2 * exp_neg(-fma(q, ih2, om * dt), tab);
                    v[3] += e;
                    v[4] = fma(e, dt, v[4]);
                    v[5] = fma(e, q, v[5]);
                }
            add();
            ne = 0;
            __syncwarp();
        };

        const int64_t jb = sg * seg, je = min(jb + seg, n);
        for (int64_t j0 = jb; j0 < je; j0 += 32) {
            const int64_t jc = min(j0 + lane, n - 1);
            w.col[lane] = make_float4(bound_coord(d.x[jc] - x0), bound_coord(d.y[jc] - y0),
                                      bound_coord(d.t[jc] - t0),
                                      bound_scale(model1 ? ih2 : ih2 * d.is2[jc]));
            __syncwarp();
            const int nc = static_cast<int>(min(je - j0, static_cast<int64_t>(32)));
            for (int c = 0; c < nc; ++c) {
                const float4 q = w.col[c];
                const int j = static_cast<int>(j0) + c;
                const float dx = low_diff(xf, q.x), dy = low_diff(yf, q.y), dt = low_diff(tf, q.z);
                const float r2 = fmaf(dx, dx, dy * dy);
                // (negated: a NaN bound keeps the pair)
                if ((j < lo || j >= hi) && !(fmaf(r2, ix2f, dt * dt * it2f) > R64_ZERO)) w.qb[nb++][lane] = j;
                if (j < lo && !(fmaf(r2, q.w, omf * dt) > R64_ZERO)) w.qe[ne++][lane] = j;
                if (__any_sync(ALL, nb == R64_QB)) {
                    __syncwarp();
                    eval_b();
                }
                if (__any_sync(ALL, ne == R64_QE)) {
                    __syncwarp();
                    eval_e();
                }
            }
            __syncwarp();
        }
        __syncwarp();
        eval_b();
        eval_e();
        if (live)
            for (int q = 0; q < 6; ++q) out[(static_cast<int64_t>(sg) * 6 + q) * stride + i - origin] = total[q] + v[q];
    }
}

// Column segments per row group: up to 32, for four items per warp of a full
// chip, so that few rows still fill it and uneven items even out (N = 2,000: 63
// groups x 32).  More than one segment needs at most rows64_scratch doubles for
// the partial sums of any rows of n events: 1.5 KB an event, up to 7.5 MB (152 SMs).
int rows64_segments(int64_t rows, int sms) {
    const int64_t groups = (rows + 31) / 32, s = 4ll * R64_WARPS * sms / groups;
    return static_cast<int>(std::min<int64_t>(std::max<int64_t>(s, 1), 32));
}
size_t rows64_scratch(int64_t n, int sms) {
    const int64_t groups = (n + 31) / 32;
    return static_cast<size_t>(std::min<int64_t>(32 * groups, 4ll * R64_WARPS * sms)) * 32 * 6;
}

// Rows [rb, re) into out (one segment: the accumulators, [6][npad]; else the
// scratch, [segment][6][rows rounded up to 32]); ctr[CT_WORK] must be zero.
cudaError_t launch_pairs64(const hawkes_ctx* c, bool model1, bool bgt, int64_t rb, int64_t re, double* out) {
    const int segments = rows64_segments(re - rb, c->sms);
    const int groups = static_cast<int>((re - rb + 31) / 32);
    const int64_t items = static_cast<int64_t>(groups) * segments;
    const int warps = static_cast<int>(std::min<int64_t>((items + c->sms - 1) / c->sms, R64_WARPS));
    const int grid = static_cast<int>(std::min<int64_t>((items + warps - 1) / warps, c->sms));
    const size_t smem = std::max(EXP_N * sizeof(double2) + warps * sizeof(R64Warp), spread_smem(grid, c->sms));
    return launch_chained(bgt ? k_pairs64<true> : k_pairs64<false>, grid, 32 * warps, smem, c->stream, eval_desc(c),
                          model1 ? 1 : 0, rb, re, groups, segments, out,
                          segments > 1 ? static_cast<int64_t>(groups) * 32 : c->npad, segments > 1 ? rb : 0);
}

cudaError_t pairs64_setup_attributes() {
    for (auto* k : {k_pairs64<false>, k_pairs64<true>}) {
        const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   static_cast<int>(spread_smem(1, 1)));
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace hk

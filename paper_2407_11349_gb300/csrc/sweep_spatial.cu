// Exact spatial skip of the pair sweep (flag HAWKES_SKIP_SPATIAL).
//
// At the sizes of the paper most pair terms are exact FP32 zeros because the
// two events are far apart: a background term B' = 2^-(dt~^2 + r~^2) flushes
// to zero once its exponent passes 126, and an excitation term once
// omega~ dt~ + beta r~^2 - ce passes 126 (ex2.approx.ftz).  This path orders
// the events so that neighbours in the order are neighbours in space and time,
// and evaluates, for each group of 32 rows, only the columns that can hold a
// nonzero term:
//   - Order (host, on first use): time windows of about `window` events, each
//     split by a k-d tree over (x, y, t) down to chunks of 32 events (tiles of
//     256).  Space and time are weighed by tau_x and tau_t of the call that
//     builds the order.  Locations that will be redrawn inside their counties
//     say little beyond the county, so they enter as the county's mean plus a
//     fifth of the offset from it.
//   - Per call: records in that order and the bounding box, time range and
//     largest excitation reach of every chunk and tile (a resample moves them
//     with the events).
//   - Sweep: one warp per group of 32 rows (one chunk of the order, a row per
//     lane).  It tests tiles, then chunks, against its rows' box, then the
//     chunk's 32 events, one per lane, and appends the survivors to two small
//     buffers in shared memory (background, excitation).  A full buffer is
//     evaluated, two columns per packed f32x2 register.
// Every test keeps 2 units of margin on the base-2 exponent, and the boxes are
// widened by the FP32 rounding of the coordinates, so what is left out is an
// exact FP32 zero; the rest is the full sweep's sum in another order.
//
// What bounds it: shared-memory reads (a column's 24 bytes go to every lane;
// 74% of the wavefronts) and instruction issue (67%) in the evaluation of the
// columns that pass the point test; the FP32 pipe is 46% busy.  Two rows per
// lane would halve the reads, but the box of 64 rows keeps 48% more columns.
// At N = 1,000,000 (3,143 counties, 1,200 days) a row has 1,811
// columns with a nonzero background and 14 with a nonzero excitation; point
// tests against the box of 32 rows leave 4,070 and 1,210, in 4.1 ms.  (The former
// design, 256 x 256 tile pairs kept whole by box tests and swept through
// shared-memory tiles, left about 40,000 with both terms: 45 ms.)
// Tie and causality indicators come from each event's index in the time order,
// carried beside its record, and are only tested for columns that can share a
// time with the rows.  Row sums go to the FP64 accumulators of the events'
// original indices; finalisation is shared with the other paths.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <system_error>
#include <thread>
#include <vector>

#include "sweep_kernel.cuh"

namespace hk {

constexpr int SP_CH = 32;              // events per chunk: a row group, and the finest column unit
constexpr int SP_WARPS = 8, SP_THREADS = 32 * SP_WARPS;
// Resident CTAs per SM.  At N = 1,000,000: 2 4.30 ms, 3 4.07, 4 (64 registers,
// spills) 4.52, 5 6.3.
constexpr int SP_BPSM = 3;
constexpr int SP_BUF = 64;             // buffered columns (32 evaluated at a time)
constexpr int SP_LIST = 128;           // chunks listed before they are read
constexpr int SP_B_PLANES = 7, SP_E_PLANES = 9;
constexpr int32_t SP_TIED = 1 << 30;   // flag in a position's rank: other events share the time
constexpr float SP_ZERO = 128.f;       // exponent beyond which a term counts as zero (126 + margin)
static_assert(NPAD_MULT % TC == 0 && TC == 8 * SP_CH, "a tile is 8 chunks");

struct SpatialState {
    int64_t window = 131072;  // target events per time window
    bool built = false;
    int ntiles = 0;           // npad / TC
    int32_t* rank = nullptr;  // [npad] time-order index at each position, | SP_TIED (-1: padding)
    float4* meta = nullptr;   // [2 x chunks], then [2 x tiles]: SpBox of each
};

void spatial_free(hawkes_ctx* c) {
    if (!c->sp) return;
    SpatialState* s = c->sp;
    if (s->rank) cudaFree(s->rank);
    if (s->meta) cudaFree(s->meta);
    delete s;
    c->sp = nullptr;
}

void spatial_invalidate(hawkes_ctx* c) {
    if (c->sp) c->sp->built = false;
}

int spatial_set_window(hawkes_ctx* c, int64_t window) {
    if (window < TC) return HAWKES_ERR_ARG;
    if (!c->sp) {
        c->sp = new (std::nothrow) SpatialState();
        if (!c->sp) return HAWKES_ERR_OOM;
    }
    if (c->sp->window != window) {
        c->sp->window = window;
        c->sp->built = false;
    }
    return HAWKES_OK;
}

// Split [a, b) of the permutation at medians of its widest side, down to
// chunks; parts stay whole tiles while larger than a tile.
struct SpPoint {
    float c[3];
    int32_t e;
};
static void sp_split(SpPoint* a, SpPoint* b) {
    while (b - a > SP_CH) {
        const int64_t len = b - a, unit = len > TC ? TC : SP_CH;
        float lo[3], hi[3];
        for (int k = 0; k < 3; ++k) lo[k] = hi[k] = a->c[k];
        for (const SpPoint* p = a + 1; p < b; ++p)
            for (int k = 0; k < 3; ++k) {
                lo[k] = std::min(lo[k], p->c[k]);
                hi[k] = std::max(hi[k], p->c[k]);
            }
        int ax = 0;
        for (int k = 1; k < 3; ++k)
            if (hi[k] - lo[k] > hi[ax] - lo[ax]) ax = k;
        SpPoint* m = a + std::min((len / 2 + unit - 1) / unit * unit, (len - 1) / unit * unit);
        std::nth_element(a, m, b, [ax](const SpPoint& u, const SpPoint& v) {
            return u.c[ax] < v.c[ax] || (u.c[ax] == v.c[ax] && u.e < v.e);
        });
        sp_split(m, b);
        b = m;
    }
}

static int build_order(hawkes_ctx* c, double tau_x, double tau_t) {
    SpatialState* sp = c->sp;
    const int64_t n = c->n, npad = c->npad;
    std::vector<double> t(n), x(n), y(n);
    std::vector<int32_t> cty(n), lo(n), hi(n);
    if (cudaStreamSynchronize(c->stream) != cudaSuccess ||
        cudaMemcpy(t.data(), c->t, n * sizeof(double), cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemcpy(x.data(), c->x, n * sizeof(double), cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemcpy(y.data(), c->y, n * sizeof(double), cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemcpy(cty.data(), c->county, n * sizeof(int32_t), cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemcpy(lo.data(), c->lo, n * sizeof(int32_t), cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemcpy(hi.data(), c->hi, n * sizeof(int32_t), cudaMemcpyDeviceToHost) != cudaSuccess)
        return HAWKES_ERR_CUDA;
    if (c->counties_ok) {  // a resample can move the events inside their counties
        std::vector<double> mx(c->n_counties, 0.0), my(c->n_counties, 0.0), cnt(c->n_counties, 0.0);
        for (int64_t i = 0; i < n; ++i) {
            mx[cty[i]] += x[i];
            my[cty[i]] += y[i];
            cnt[cty[i]] += 1.0;
        }
        for (int64_t i = 0; i < n; ++i) {
            const double cx = mx[cty[i]] / cnt[cty[i]], cy = my[cty[i]] / cnt[cty[i]];
            x[i] = cx + 0.2 * (x[i] - cx);
            y[i] = cy + 0.2 * (y[i] - cy);
        }
    }
    std::vector<SpPoint> pt(n);
    for (int64_t i = 0; i < n; ++i)
        pt[i] = SpPoint{{static_cast<float>((x[i] - x[0]) / tau_x), static_cast<float>((y[i] - y[0]) / tau_x),
                         static_cast<float>((t[i] - t[0]) / tau_t)},
                        static_cast<int32_t>(i)};
    // time windows (whole tiles), split independently on a few host threads
    const int64_t w = (sp->window + TC - 1) / TC * TC;
    const int64_t nw = (n + w - 1) / w;
    auto work = [&](int64_t k0, int64_t step) {
        for (int64_t k = k0; k < nw; k += step) sp_split(pt.data() + k * w, pt.data() + std::min(n, (k + 1) * w));
    };
    const int64_t nth = std::min<int64_t>(nw, n > 50000 ? 8 : 1);
    std::vector<std::thread> th;
    int64_t started = 1;  // this thread takes window 0, nth, 2 nth, ...
    try {
        for (; started < nth; ++started) th.emplace_back(work, started, nth);
    } catch (const std::system_error&) {  // no more threads: the rest runs here
    }
    work(0, nth);
    for (int64_t k = started; k < nth; ++k) work(k, nth);
    for (std::thread& q : th) q.join();
    std::vector<int32_t> rank(npad, -1);
    for (int64_t p = 0; p < n; ++p) {
        const int32_t e = pt[p].e;
        rank[p] = hi[e] - lo[e] > 1 ? (e | SP_TIED) : e;
    }
    const int ntiles = static_cast<int>(npad / TC);
    if (sp->ntiles != ntiles || !sp->rank || !sp->meta) {
        if (sp->rank) cudaFree(sp->rank);
        if (sp->meta) cudaFree(sp->meta);
        sp->rank = nullptr;
        sp->meta = nullptr;
        if (cudaMalloc(&sp->rank, npad * sizeof(int32_t)) != cudaSuccess ||
            cudaMalloc(&sp->meta, 2 * static_cast<size_t>(9 * ntiles) * sizeof(float4)) != cudaSuccess) {
            cudaGetLastError();
            return HAWKES_ERR_OOM;
        }
        sp->ntiles = ntiles;
    }
    if (cudaMemcpy(sp->rank, rank.data(), npad * sizeof(int32_t), cudaMemcpyHostToDevice) != cudaSuccess)
        return HAWKES_ERR_CUDA;
    sp->built = true;
    return HAWKES_OK;
}

// Build the order from the current events (synchronous; the locations used for
// the order are the current ones).  p: the call's parameters on the host, or
// null with d_p on the device; they only weigh space against time.
int spatial_build(hawkes_ctx* c, const hawkes_params* p, const hawkes_params* d_p) {
    if (!c->sp) {
        const int rc = spatial_set_window(c, 131072);
        if (rc != HAWKES_OK) return rc;
    }
    if (c->sp->built) return HAWKES_OK;
    if (c->n >= SP_TIED) return HAWKES_ERR_ARG;
    hawkes_params q{};
    if (p)
        q = *p;
    else if (cudaStreamSynchronize(c->stream) != cudaSuccess ||
             cudaMemcpy(&q, d_p, sizeof(q), cudaMemcpyDeviceToHost) != cudaSuccess)
        return HAWKES_ERR_CUDA;
    auto usable = [](double v) { return v > 1e-30 && v < 1e30; };
    if (!usable(q.tau_x) || !usable(q.tau_t)) q.tau_x = q.tau_t = 1.0;
    try {
        return build_order(c, q.tau_x, q.tau_t);
    } catch (const std::bad_alloc&) {
        return HAWKES_ERR_OOM;
    }
}

// Bounds of a set of events, in scaled units: box, time range, largest ce,
// smallest beta.  Empty: x0 > x1.
struct SpBox {
    float x0, x1, y0, y1, t0, t1, ce, beta;
};

__device__ __forceinline__ SpBox sp_load(const float4* __restrict__ meta, int k) {
    const float4 a = meta[2 * k], b = meta[2 * k + 1];
    return SpBox{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
}
__device__ __forceinline__ void sp_store(float4* meta, int k, const SpBox& v) {
    meta[2 * k] = make_float4(v.x0, v.x1, v.y0, v.y1);
    meta[2 * k + 1] = make_float4(v.t0, v.t1, v.ce, v.beta);
}
__device__ __forceinline__ SpBox sp_empty() {
    return SpBox{1e30f, -1e30f, 1e30f, -1e30f, 1e30f, -1e30f, -1e30f, 1e30f};
}
__device__ __forceinline__ void sp_join(SpBox& a, const SpBox& b) {
    a.x0 = fminf(a.x0, b.x0); a.x1 = fmaxf(a.x1, b.x1);
    a.y0 = fminf(a.y0, b.y0); a.y1 = fmaxf(a.y1, b.y1);
    a.t0 = fminf(a.t0, b.t0); a.t1 = fmaxf(a.t1, b.t1);
    a.ce = fmaxf(a.ce, b.ce); a.beta = fminf(a.beta, b.beta);
}
// Widen [lo, hi] by 2^-22 of its magnitude: more than the rounding to FP32 of
// its own ends and of any point compared with it nearby.
__device__ __forceinline__ void sp_widen(float& lo, float& hi) {
    const float s = 2.384185791015625e-07f * fmaxf(fabsf(lo), fabsf(hi));
    lo -= s;
    hi += s;
}

// Stage the records in the spatial order (negated column values): planes
// ra[npad] = (-x hi, -x lo, -y hi, -y lo), rb[npad] = (-t hi, -t lo, -beta, ce),
// with t~ = (t - t_1) sqrt(a_t) in two FP32 words like the coordinates, and
// the boxes of the chunks and tiles (one block per tile).
__global__ void __launch_bounds__(TC) k_sp_prep(EvalDesc d, const int32_t* __restrict__ rank, int model1,
                                                float4* __restrict__ ra, float4* __restrict__ rb,
                                                float4* __restrict__ meta, int ntiles) {
    if (d.cc[CC_VALID] == 0.0) return;
    const double kx = d.cc[CC_KX], kt = d.cc[CC_KT], tf = d.t[0];
    const double beta0 = (d.cc[CC_TX] * d.cc[CC_TX]) / (d.cc[CC_H] * d.cc[CC_H]);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __shared__ SpBox boxes[TC / SP_CH];
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int64_t p = static_cast<int64_t>(tile) * TC + threadIdx.x;
        const int32_t r = rank[p];
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = make_float4(-PAD_T, 0.f, 0.f, -1e30f);
        SpBox box = sp_empty();
        if (r >= 0) {
            const int32_t e = r & ~SP_TIED;
            const double ts = (d.t[e] - tf) * kt, xs = d.x[e] * kx, ys = d.y[e] * kx;
            const float th = static_cast<float>(ts), xh = static_cast<float>(xs), yh = static_cast<float>(ys);
            const float beta = static_cast<float>(model1 ? beta0 : beta0 * d.is2[e]);
            const float ce = model1 ? 0.f : d.ce[e];
            a = make_float4(-xh, -static_cast<float>(xs - static_cast<double>(xh)), -yh,
                            -static_cast<float>(ys - static_cast<double>(yh)));
            b = make_float4(-th, -static_cast<float>(ts - static_cast<double>(th)), -beta, ce);
            box = SpBox{xh, xh, yh, yh, th, th, ce, beta};
        }
        ra[p] = a;
        rb[p] = b;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            SpBox q;
            q.x0 = __shfl_xor_sync(0xffffffffu, box.x0, o); q.x1 = __shfl_xor_sync(0xffffffffu, box.x1, o);
            q.y0 = __shfl_xor_sync(0xffffffffu, box.y0, o); q.y1 = __shfl_xor_sync(0xffffffffu, box.y1, o);
            q.t0 = __shfl_xor_sync(0xffffffffu, box.t0, o); q.t1 = __shfl_xor_sync(0xffffffffu, box.t1, o);
            q.ce = __shfl_xor_sync(0xffffffffu, box.ce, o); q.beta = __shfl_xor_sync(0xffffffffu, box.beta, o);
            sp_join(box, q);
        }
        if (lane == 0) {
            if (box.x0 <= box.x1) {
                sp_widen(box.x0, box.x1);
                sp_widen(box.y0, box.y1);
                sp_widen(box.t0, box.t1);
            }
            boxes[warp] = box;
            sp_store(meta, tile * (TC / SP_CH) + warp, box);
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int k = 1; k < TC / SP_CH; ++k) sp_join(box, boxes[k]);
            sp_store(meta, ntiles * (TC / SP_CH) + tile, box);
        }
        __syncthreads();
    }
}

struct SpArgs {
    const float4* ra;
    const float4* rb;
    const int32_t* rank;
    const int32_t* lo;
    const int32_t* hi;
    const double* cc;
    double* acc;
    const float4* cmeta;
    const float4* tmeta;
    int64_t npad;
    int ntiles, groups, parts;
};

// Can a column of box (or point) c hold a nonzero background / excitation term
// for some row of box w?
__device__ __forceinline__ float sp_gap(float lo, float hi, float a0, float a1) {
    return fmaxf(0.f, fmaxf(a0 - hi, lo - a1));
}
__device__ __forceinline__ void sp_near(const SpBox& w, const SpBox& c, float omt, bool& nb, bool& ne) {
    const float dx = sp_gap(w.x0, w.x1, c.x0, c.x1), dy = sp_gap(w.y0, w.y1, c.y0, c.y1);
    const float r2 = fmaf(dx, dx, dy * dy), g = sp_gap(w.t0, w.t1, c.t0, c.t1);
    nb = !(fmaf(g, g, r2) > SP_ZERO);  // (negated: a NaN is kept, and reported as ever)
    ne = c.t0 <= w.t1 && !(c.ce - omt * fmaxf(0.f, w.t0 - c.t1) - c.beta * r2 < -SP_ZERO);
}

// A lane's row (values doubled for packed arithmetic) and its sums over the
// even and odd columns.
struct SpRow {
    float2 th, tl, xh, xl, yh, yl;
    float2 sB, sBr, sBt, sE, sEt, sEq;
    int lo, hi;
};

__device__ __forceinline__ float2 half4(const float4& v, int h) { return h ? f2(v.z, v.w) : f2(v.x, v.y); }

// Background of `quads` x 4 buffered columns against the lane's row.
template <bool MASK, bool LL>
__device__ __forceinline__ void sp_eval_b(const float* __restrict__ buf, int quads, SpRow& w) {
#pragma unroll 4
    for (int q = 0; q < quads; ++q) {
        const float4* p = reinterpret_cast<const float4*>(buf) + q;
        const float4 xh = p[0 * SP_BUF / 4], xl = p[1 * SP_BUF / 4], yh = p[2 * SP_BUF / 4],
                     yl = p[3 * SP_BUF / 4], th = p[4 * SP_BUF / 4], tl = p[5 * SP_BUF / 4];
        int4 rk;
        if (MASK) rk = *reinterpret_cast<const int4*>(p + 6 * SP_BUF / 4);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float2 dt = add2(add2(w.th, half4(th, h)), add2(w.tl, half4(tl, h)));
            const float2 dx = add2(add2(w.xh, half4(xh, h)), add2(w.xl, half4(xl, h)));
            const float2 dy = add2(add2(w.yh, half4(yh, h)), add2(w.yl, half4(yl, h)));
            const float2 r2 = fma2(dy, dy, mul2(dx, dx));
            const float2 dt2 = mul2(dt, dt);
            const float2 aB = add2(dt2, r2);
            float2 B = f2(ex2(-aB.x), ex2(-aB.y));
            if (MASK) {  // t_j != t_i
                const int r0 = h ? rk.z : rk.x, r1 = h ? rk.w : rk.y;
                B.x = (r0 < w.lo || r0 >= w.hi) ? B.x : 0.f;
                B.y = (r1 < w.lo || r1 >= w.hi) ? B.y : 0.f;
            }
            w.sB = add2(w.sB, B);
            if (!LL) {
                w.sBr = fma2(B, r2, w.sBr);
                w.sBt = fma2(B, dt2, w.sBt);
            }
        }
    }
}

// Excitation of `quads` x 4 buffered columns (planes as above, then -beta, ce).
template <bool MASK, bool LL>
__device__ __forceinline__ void sp_eval_e(const float* __restrict__ buf, int quads, float2 nomt, SpRow& w) {
#pragma unroll 1
    for (int q = 0; q < quads; ++q) {
        const float4* p = reinterpret_cast<const float4*>(buf) + q;
        const float4 xh = p[0 * SP_BUF / 4], xl = p[1 * SP_BUF / 4], yh = p[2 * SP_BUF / 4],
                     yl = p[3 * SP_BUF / 4], th = p[4 * SP_BUF / 4], tl = p[5 * SP_BUF / 4],
                     nb = p[7 * SP_BUF / 4], ce = p[8 * SP_BUF / 4];
        int4 rk;
        if (MASK) rk = *reinterpret_cast<const int4*>(p + 6 * SP_BUF / 4);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float2 dt = add2(add2(w.th, half4(th, h)), add2(w.tl, half4(tl, h)));
            const float2 dx = add2(add2(w.xh, half4(xh, h)), add2(w.xl, half4(xl, h)));
            const float2 dy = add2(add2(w.yh, half4(yh, h)), add2(w.yl, half4(yl, h)));
            const float2 r2 = fma2(dy, dy, mul2(dx, dx));
            const float2 nv = mul2(half4(nb, h), r2);
            const float2 arg = add2(fma2(nomt, dt, nv), half4(ce, h));
            float2 E = f2(ex2(arg.x), ex2(arg.y));
            if (MASK) {  // t_j < t_i
                const int r0 = h ? rk.z : rk.x, r1 = h ? rk.w : rk.y;
                E.x = r0 < w.lo ? E.x : 0.f;
                E.y = r1 < w.lo ? E.y : 0.f;
            }
            w.sE = add2(w.sE, E);
            if (!LL) {
                w.sEt = fma2(E, dt, w.sEt);
                w.sEq = fma2(E, nv, w.sEq);
            }
        }
    }
}

// Shared memory of a warp: the two column buffers and the chunk list.
struct SpWarp {
    float b[SP_B_PLANES * SP_BUF];
    float e[SP_E_PLANES * SP_BUF];
    int list[SP_LIST];
};

// Persistent warps over items (row group, part of the column tiles).
template <bool LL>
__global__ void __launch_bounds__(SP_THREADS, SP_BPSM) k_sweep_sp(SpArgs a, int* __restrict__ ctr, int nitems) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31;
    SpWarp& sw = reinterpret_cast<SpWarp*>(smem)[threadIdx.x >> 5];
    const double* cc = a.cc;
    if (cc[CC_VALID] == 0.0) return;
    const float omt = static_cast<float>(cc[CC_OMT]);
    const float2 nomt = f2(-omt, -omt);
    const unsigned below = (1u << lane) - 1u;
    constexpr unsigned ALL = 0xffffffffu;

    for (;;) {
        int item = 0;
        if (lane == 0) item = atomicAdd(ctr + CT_WORK, 1);
        item = __shfl_sync(ALL, item, 0);
        if (item >= nitems) return;
        const int g = item / a.parts, part = item % a.parts;
        const int64_t p0 = static_cast<int64_t>(g) * SP_CH;
        const SpBox box = sp_load(a.cmeta, g);
        if (!(box.x0 <= box.x1)) continue;  // padding only
        SpRow w;
        const int rr = a.rank[p0 + lane];
        const int e = rr >= 0 ? rr & ~SP_TIED : -1;
        {
            const float4 qa = a.ra[p0 + lane], qb = a.rb[p0 + lane];
            w.xh = f2(-qa.x, -qa.x); w.xl = f2(-qa.y, -qa.y);
            w.yh = f2(-qa.z, -qa.z); w.yl = f2(-qa.w, -qa.w);
            w.th = f2(-qb.x, -qb.x); w.tl = f2(-qb.y, -qb.y);
        }
        w.lo = e >= 0 ? a.lo[e] : 0;
        w.hi = e >= 0 ? a.hi[e] : 0;
        w.sB = w.sBr = w.sBt = w.sE = w.sEt = w.sEq = f2(0.f, 0.f);
        // time-order indices that some row must be compared with one by one
        const int lo_min = __reduce_min_sync(ALL, e >= 0 ? w.lo : 0x7fffffff);
        const int hi_max = __reduce_max_sync(ALL, e >= 0 ? w.hi : 0);

        int nB = 0, nE = 0;            // buffered columns
        bool maskB = false, maskE = false;
        int tile0 = 0;                 // next round of 32 tiles (of this part)
        unsigned mT = 0;               // surviving tiles of the current round
        int nlist = 0;
        for (;;) {
            // list chunks that can hold a nonzero term
            while (nlist <= SP_LIST - 32) {
                if (mT == 0) {
                    const int first = tile0 * a.parts + part;
                    if (first >= a.ntiles) break;
                    const int t = (tile0 + lane) * a.parts + part;
                    bool nb = false, ne = false;
                    if (t < a.ntiles) sp_near(box, sp_load(a.tmeta, t), omt, nb, ne);
                    mT = __ballot_sync(ALL, nb || ne);
                    if (mT == 0) tile0 += 32;
                    continue;
                }
                // the 8 chunks of the next (up to) 4 surviving tiles
                unsigned m = mT;
                for (int k = 0; k < 4; ++k) mT &= mT - 1;
                for (int k = 0; k < (lane >> 3); ++k) m &= m - 1;
                const bool has = m != 0;
                const int t = has ? (tile0 + __ffs(m) - 1) * a.parts + part : 0;
                const int ch = t * (TC / SP_CH) + (lane & 7);
                bool nb = false, ne = false;
                if (has) sp_near(box, sp_load(a.cmeta, ch), omt, nb, ne);
                const unsigned keep = __ballot_sync(ALL, nb || ne);
                if (nb || ne) sw.list[nlist + __popc(keep & below)] = ch | (nb ? 1 << 29 : 0) | (ne ? 1 << 30 : 0);
                nlist += __popc(keep);
                if (mT == 0) tile0 += 32;
            }
            __syncwarp();
            if (nlist == 0) break;
            // read the listed chunks, one event per lane, the next one ahead
            int cur = sw.list[0];
            int64_t p = static_cast<int64_t>(cur & ((1 << 29) - 1)) * SP_CH + lane;
            float4 qa = a.ra[p], qb = a.rb[p];
            int rk = a.rank[p];
            for (int k = 0; k < nlist; ++k) {
                const int id = cur;
                const float4 ca = qa, cb = qb;
                const int rank = rk & ~SP_TIED;
                const bool real = rk >= 0;
                const bool tied = (rk & SP_TIED) != 0 || (id & ((1 << 29) - 1)) == g;
                if (k + 1 < nlist) {
                    cur = sw.list[k + 1];
                    p = static_cast<int64_t>(cur & ((1 << 29) - 1)) * SP_CH + lane;
                    qa = a.ra[p];
                    qb = a.rb[p];
                    rk = a.rank[p];
                }
                const float dx = sp_gap(box.x0, box.x1, -ca.x, -ca.x), dy = sp_gap(box.y0, box.y1, -ca.z, -ca.z);
                const float r2 = fmaf(dx, dx, dy * dy);
                if (id & (1 << 29)) {
                    const float gap = sp_gap(box.t0, box.t1, -cb.x, -cb.x);
                    const bool keep = real && !(fmaf(gap, gap, r2) > SP_ZERO);
                    const unsigned bal = __ballot_sync(ALL, keep);
                    maskB |= __any_sync(ALL, keep && tied && rank >= lo_min && rank < hi_max);
                    if (keep) {
                        float* b = sw.b + nB + __popc(bal & below);
                        b[0 * SP_BUF] = ca.x; b[1 * SP_BUF] = ca.y; b[2 * SP_BUF] = ca.z; b[3 * SP_BUF] = ca.w;
                        b[4 * SP_BUF] = cb.x; b[5 * SP_BUF] = cb.y; b[6 * SP_BUF] = __int_as_float(rank);
                    }
                    nB += __popc(bal);
                    if (nB >= 32) {
                        __syncwarp();
                        if (maskB) sp_eval_b<true, LL>(sw.b, 8, w);
                        else sp_eval_b<false, LL>(sw.b, 8, w);
                        nB -= 32;
                        maskB = maskB && nB > 0;
                        __syncwarp();
                        if (lane < nB)
#pragma unroll
                            for (int q = 0; q < SP_B_PLANES; ++q) sw.b[q * SP_BUF + lane] = sw.b[q * SP_BUF + 32 + lane];
                        __syncwarp();
                    }
                }
                if (id & (1 << 30)) {
                    const float tj = -cb.x;
                    const bool keep = real && tj <= box.t1 &&
                                      !(cb.w - omt * fmaxf(0.f, box.t0 - tj) + cb.z * r2 < -SP_ZERO);
                    const unsigned bal = __ballot_sync(ALL, keep);
                    maskE |= __any_sync(ALL, keep && rank >= lo_min);
                    if (keep) {
                        float* b = sw.e + nE + __popc(bal & below);
                        b[0 * SP_BUF] = ca.x; b[1 * SP_BUF] = ca.y; b[2 * SP_BUF] = ca.z; b[3 * SP_BUF] = ca.w;
                        b[4 * SP_BUF] = cb.x; b[5 * SP_BUF] = cb.y; b[6 * SP_BUF] = __int_as_float(rank);
                        b[7 * SP_BUF] = cb.z; b[8 * SP_BUF] = cb.w;
                    }
                    nE += __popc(bal);
                    if (nE >= 32) {
                        __syncwarp();
                        if (maskE) sp_eval_e<true, LL>(sw.e, 8, nomt, w);
                        else sp_eval_e<false, LL>(sw.e, 8, nomt, w);
                        nE -= 32;
                        maskE = maskE && nE > 0;
                        __syncwarp();
                        if (lane < nE)
#pragma unroll
                            for (int q = 0; q < SP_E_PLANES; ++q) sw.e[q * SP_BUF + lane] = sw.e[q * SP_BUF + 32 + lane];
                        __syncwarp();
                    }
                }
            }
            nlist = 0;
            __syncwarp();
        }
        // what is left in the buffers, filled up to quads with columns whose
        // terms are zero
        const int qB = (nB + 3) >> 2, qE = (nE + 3) >> 2;
        if (nB + lane < 4 * qB) {
            for (int q = 0; q < SP_B_PLANES; ++q) sw.b[q * SP_BUF + nB + lane] = 0.f;
            sw.b[4 * SP_BUF + nB + lane] = -PAD_T;
        }
        if (nE + lane < 4 * qE) {
            for (int q = 0; q < SP_E_PLANES; ++q) sw.e[q * SP_BUF + nE + lane] = 0.f;
            sw.e[8 * SP_BUF + nE + lane] = -1e30f;
        }
        __syncwarp();
        if (maskB) sp_eval_b<true, LL>(sw.b, qB, w);
        else sp_eval_b<false, LL>(sw.b, qB, w);
        if (maskE) sp_eval_e<true, LL>(sw.e, qE, nomt, w);
        else sp_eval_e<false, LL>(sw.e, qE, nomt, w);
        __syncwarp();
        if (e >= 0) {
            const float v[6] = {w.sB.x + w.sB.y, w.sBr.x + w.sBr.y, w.sBt.x + w.sBt.y,
                                w.sE.x + w.sE.y, w.sEt.x + w.sEt.y, w.sEq.x + w.sEq.y};
            double* acc = a.acc + e;
            if (v[0] != 0.f) atomicAdd(acc, static_cast<double>(v[0]));
            if (v[3] != 0.f) atomicAdd(acc + 3 * a.npad, static_cast<double>(v[3]));
            if (!LL) {
                if (v[1] != 0.f) atomicAdd(acc + 1 * a.npad, static_cast<double>(v[1]) * cc[CC_SR]);
                if (v[2] != 0.f) atomicAdd(acc + 2 * a.npad, static_cast<double>(v[2]) * cc[CC_ST]);
                if (v[4] != 0.f) atomicAdd(acc + 4 * a.npad, static_cast<double>(v[4]) * cc[CC_SET]);
                if (v[5] != 0.f) atomicAdd(acc + 5 * a.npad, -static_cast<double>(v[5]) * cc[CC_SEQ]);
            }
        }
    }
}

// Queue the spatial path's staging and sweep (after k_prep has written the
// per-call constants and zeroed the accumulators).  The records take the place
// of the staged records of the other paths.
cudaError_t spatial_launch(hawkes_ctx* c, int model1, int llonly) {
    SpatialState* sp = c->sp;
    float4* ra = reinterpret_cast<float4*>(c->rec);
    float4* rb = ra + c->npad;
    k_sp_prep<<<std::min(sp->ntiles, 8 * c->sms), TC, 0, c->stream>>>(eval_desc(c), sp->rank, model1, ra, rb,
                                                                      sp->meta, sp->ntiles);
    SpArgs a;
    a.ra = ra; a.rb = rb; a.rank = sp->rank; a.lo = c->lo; a.hi = c->hi; a.cc = c->cc; a.acc = c->acc;
    a.cmeta = sp->meta;
    a.tmeta = sp->meta + 2 * static_cast<size_t>(sp->ntiles) * (TC / SP_CH);
    a.npad = c->npad;
    a.ntiles = sp->ntiles;
    a.groups = static_cast<int>((c->n + SP_CH - 1) / SP_CH);
    // Few rows: several warps share a group's columns, until there are a
    // resident CTA's worth of warps for every SM.
    const size_t smem = SP_WARPS * sizeof(SpWarp);
    auto* kern = llonly ? k_sweep_sp<true> : k_sweep_sp<false>;
    static_assert(SP_WARPS * sizeof(SpWarp) <= 48 * 1024, "below the default dynamic limit");
    a.parts = 1;
    while (a.parts < 64 && 2 * a.parts <= a.ntiles &&
           static_cast<int64_t>(a.groups) * a.parts < static_cast<int64_t>(c->sms) * SP_BPSM * SP_WARPS)
        a.parts *= 2;
    const int64_t nitems = static_cast<int64_t>(a.groups) * a.parts;
    const int grid = static_cast<int>(std::min<int64_t>((nitems + SP_WARPS - 1) / SP_WARPS,
                                                        static_cast<int64_t>(c->sms) * SP_BPSM));
    kern<<<grid, SP_THREADS, smem, c->stream>>>(a, c->ctr, static_cast<int>(nitems));
    return cudaGetLastError();
}

}  // namespace hk

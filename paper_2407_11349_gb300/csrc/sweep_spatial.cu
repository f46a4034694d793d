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
//   - Per call: records in that order, relative to their chunk's centre, and the
//     bounding box, time range and largest excitation reach of every chunk, tile
//     and block of 32 tiles (a resample moves them with the events).
//   - Sweep: one warp per group of 32 rows (one chunk of the order, a row per
//     lane).  It tests blocks, tiles and chunks against its rows' box and lists
//     the chunks that can matter, for the background and for the excitation.
//     Then it tests a listed chunk's 32 events, one per lane, and appends the
//     survivors to a buffer in shared memory; every 32 of them are evaluated, two
//     columns per packed f32x2 register.
// Every test keeps 2 units of margin on the base-2 exponent, and the boxes are
// widened by the FP32 rounding of the coordinates, so what is left out is an
// exact FP32 zero; the rest is the full sweep's sum in another order.
//
// Coordinates: two FP32 words each, rows and columns, from the centre of the rows'
// box, as in the dense sweep.  (One word for the background of row groups up to 8
// scaled units wide took 13% less time but put up to 2^-24 of the group's width
// into every difference.)
//
// What bounds it: instruction dispatch.  A packed FP32 instruction takes two
// dispatch cycles, any other one; half of the cycles go to the evaluation of the
// columns that pass the point test.  At N = 1,000,000 (3,143 counties, 1,200 days)
// after a resample, which widens the boxes, a row has 1,811 columns with a nonzero
// background and 14 with a nonzero excitation; point tests against the box of 32
// rows leave 3,770 and 620, in 3.55 to 3.85 ms.  256 x 256 tile pairs kept whole by box
// tests and swept through shared-memory tiles took 45 ms (40,000 columns with both
// terms).  Two rows per lane would halve the shared-memory reads, but the box of 64
// rows keeps 48% more columns.
// Tie and causality indicators come from each event's index in the time order,
// carried beside its record, and are only tested for columns that can share a
// time with the rows.  Row sums go to the FP64 accumulators of the events'
// original indices; finalisation is shared with the other paths.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include "spatial_bounds.h"
#include "spatial_order.h"
#include "sweep_kernel.cuh"
#include "units.cuh"

namespace hk {

constexpr int SP_WARPS = 8, SP_THREADS = 32 * SP_WARPS;
// Resident CTAs per SM.  At N = 1,000,000: 2 4.08 ms, 3 3.86, 4 (64 registers,
// spills) 3.90.
constexpr int SP_BPSM = 3;
constexpr int SP_BUF = 64;             // buffered columns (32 evaluated at a time)
constexpr int SP_LIST = 128;           // chunks listed before their events are tested
constexpr int SP_B_PLANES = 7, SP_E_PLANES = 9;
// Kept columns after which a row's FP32 sums go to FP64, so that a chain of
// additions stays below 6,200 terms (a row has two, over even and odd columns).
// A long chain of like terms drifts by a rounding bias that grows with its
// length: with bandwidths that keep every pair of 200,000 events on integer
// days, one chain to the end left the log-likelihood 4.2e-6 and the gradient
// 9.5e-5 off; folded, 2.2e-8 and 1.5e-6.  The usual bandwidths keep about 4,000
// columns of a row and seldom come here (N = 1,000,000: 1.5% of the sweep).
constexpr int SP_FOLD = 8192;
static_assert(NPAD_MULT % TC == 0 && TC == SP_TILE && TC == 8 * SP_CH, "a tile is 8 chunks");

// Boxes and centres of the order's units, one allocation: SpBox (two float4) of
// every chunk, tile and block of 32 tiles, then the chunks' centres.
constexpr int SP_TB = 32;
constexpr int sp_blocks(int ntiles) { return (ntiles + SP_TB - 1) / SP_TB; }
constexpr size_t sp_meta_f4(int ntiles) {
    return 2 * (static_cast<size_t>(9) * ntiles + sp_blocks(ntiles)) + static_cast<size_t>(8) * ntiles;
}

struct SpatialState {
    int64_t window = 131072;  // target events per time window
    bool built = false;
    int ntiles = 0;           // npad / TC
    uint32_t* rank = nullptr; // [npad] event at each position (sp_rank)
    float4* meta = nullptr;   // SpMeta's arrays
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
    std::vector<SpPoint> pt = sp_points(t, x, y, cty, c->counties_ok ? c->n_counties : 0, tau_x, tau_t);
    sp_split_windows(pt, sp->window);
    std::vector<uint32_t> rank(npad, SP_PAD);
    for (int64_t p = 0; p < n; ++p) {
        const int32_t e = pt[p].e;
        rank[p] = sp_rank(e, hi[e] - lo[e] > 1);
    }
    const int ntiles = static_cast<int>(npad / TC);
    if (sp->ntiles != ntiles || !sp->rank || !sp->meta) {
        if (sp->rank) cudaFree(sp->rank);
        if (sp->meta) cudaFree(sp->meta);
        sp->rank = nullptr;
        sp->meta = nullptr;
        if (cudaMalloc(&sp->rank, npad * sizeof(uint32_t)) != cudaSuccess ||
            cudaMalloc(&sp->meta, sp_meta_f4(ntiles) * sizeof(float4)) != cudaSuccess) {
            cudaGetLastError();
            return HAWKES_ERR_OOM;
        }
        sp->ntiles = ntiles;
    }
    if (cudaMemcpy(sp->rank, rank.data(), npad * sizeof(uint32_t), cudaMemcpyHostToDevice) != cudaSuccess)
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

__device__ __forceinline__ SpBox sp_load(const float4* __restrict__ meta, int k) {
    const float4 a = meta[2 * k], b = meta[2 * k + 1];
    return SpBox{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
}
__device__ __forceinline__ void sp_store(float4* meta, int k, const SpBox& v) {
    meta[2 * k] = make_float4(v.x0, v.x1, v.y0, v.y1);
    meta[2 * k + 1] = make_float4(v.t0, v.t1, v.ce, v.beta);
}
__device__ __forceinline__ SpBox sp_warp_join(SpBox box) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        SpBox q;
        q.x0 = __shfl_xor_sync(0xffffffffu, box.x0, o); q.x1 = __shfl_xor_sync(0xffffffffu, box.x1, o);
        q.y0 = __shfl_xor_sync(0xffffffffu, box.y0, o); q.y1 = __shfl_xor_sync(0xffffffffu, box.y1, o);
        q.t0 = __shfl_xor_sync(0xffffffffu, box.t0, o); q.t1 = __shfl_xor_sync(0xffffffffu, box.t1, o);
        q.ce = __shfl_xor_sync(0xffffffffu, box.ce, o); q.beta = __shfl_xor_sync(0xffffffffu, box.beta, o);
        sp_join(box, q);
    }
    return box;
}

// Stage the records in the spatial order: negated distances from the chunk's
// centre in two FP32 words each,
//   ra[npad] = (-x, -y, -t, rank bits), rb[npad] = (-x lo, -y lo, -t lo, -beta), rc[npad] = ce
// (the second words belong to the first ones on sp_grid's grid),
// in scaled units (t~ = (t - t_1) sqrt(a_t)), the centres, and the boxes of the
// chunks and tiles (one block per tile).
__global__ void __launch_bounds__(TC) k_sp_prep(EvalDesc d, const uint32_t* __restrict__ rank, int model1,
                                                float4* __restrict__ ra, float4* __restrict__ rb,
                                                float* __restrict__ rc, float4* __restrict__ cmeta,
                                                float4* __restrict__ tmeta, float4* __restrict__ centre,
                                                int ntiles) {
    chain_next();
    chain_wait();
    if (d.cc[CC_VALID] == 0.0) return;
    const double kx = d.cc[CC_KX], kt = d.cc[CC_KT], tf = d.t[0];
    const double beta0 = (d.cc[CC_TX] * d.cc[CC_TX]) / (d.cc[CC_H] * d.cc[CC_H]);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __shared__ SpBox boxes[TC / SP_CH];
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int64_t p = static_cast<int64_t>(tile) * TC + threadIdx.x;
        const uint32_t r = rank[p];
        float xh = 0.f, xl = 0.f, yh = 0.f, yl = 0.f, th = 0.f, tl = 0.f, beta = 0.f, ce = -1e30f;
        SpBox box = sp_empty();
        if (r != SP_PAD) {
            const int32_t e = sp_event(r);
            const double ts = (d.t[e] - tf) * kt, xs = d.x[e] * kx, ys = d.y[e] * kx;
            th = static_cast<float>(ts);
            xh = static_cast<float>(xs);
            yh = static_cast<float>(ys);
            tl = static_cast<float>(ts - static_cast<double>(th));
            xl = static_cast<float>(xs - static_cast<double>(xh));
            yl = static_cast<float>(ys - static_cast<double>(yh));
            beta = static_cast<float>(model1 ? beta0 : beta0 * d.is2[e]);
            ce = model1 ? 0.f : d.ce[e];
            box = SpBox{xh, xh, yh, yh, th, th, ce, beta};
        }
        box = sp_warp_join(box);
        const bool any = box.x0 <= box.x1;
        const float cx = any ? sp_mid(box.x0, box.x1) : 0.f, cy = any ? sp_mid(box.y0, box.y1) : 0.f,
                    ct = any ? sp_mid(box.t0, box.t1) : 0.f;
        float4 a = make_float4(0.f, 0.f, -PAD_T, __uint_as_float(SP_PAD)), b = make_float4(0.f, 0.f, 0.f, 0.f);
        if (r != SP_PAD) {
            a.w = __uint_as_float(r);
            b.w = -beta;
            sp_recentre(cx, xh, xl, a.x, b.x);
            sp_recentre(cy, yh, yl, a.y, b.y);
            sp_recentre(ct, th, tl, a.z, b.z);
        }
        ra[p] = a;
        rb[p] = b;
        rc[p] = ce;
        if (lane == 0) {
            if (any) {
                sp_widen(box.x0, box.x1);
                sp_widen(box.y0, box.y1);
                sp_widen(box.t0, box.t1);
            }
            boxes[warp] = box;
            sp_store(cmeta, tile * (TC / SP_CH) + warp, box);
            centre[tile * (TC / SP_CH) + warp] = make_float4(cx, cy, ct, 0.f);
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int k = 1; k < TC / SP_CH; ++k) sp_join(box, boxes[k]);
            sp_store(tmeta, tile, box);
        }
        __syncthreads();
    }
}

// Boxes of the blocks of 32 tiles, one warp each.
__global__ void k_sp_blocks(const float4* tmeta, float4* bmeta, int ntiles, const double* cc) {
    chain_next();
    chain_wait();
    if (cc[CC_VALID] == 0.0) return;
    const int t = blockIdx.x * SP_TB + threadIdx.x;
    const SpBox box = sp_warp_join(t < ntiles ? sp_load(tmeta, t) : sp_empty());
    if (threadIdx.x == 0) sp_store(bmeta, blockIdx.x, box);
}

struct SpArgs {
    const float4* ra;
    const float4* rb;
    const float* rc;
    const int32_t* lo;
    const int32_t* hi;
    const double* cc;
    double* acc;
    const float4* cmeta;
    const float4* tmeta;
    const float4* bmeta;
    const float4* centre;
    int64_t npad;
    int ntiles, groups, parts;
};

// A lane's row: its sums over the even and odd columns.  (Its coordinates are in
// the warp's shared memory.)
struct SpRow {
    float2 sB, sBr, sBt, sE, sEt, sEq;
    int lo, hi;
};

// Shared memory of a warp: the two column buffers, the rows' two-word
// coordinates (x hi, x lo, y hi, y lo, t hi, t lo) and the chunk list.
struct SpWarp {
    float b[SP_B_PLANES * SP_BUF];
    float e[SP_E_PLANES * SP_BUF];
    float row[6 * SP_CH];
    float4 list[SP_LIST];
};

// The differences of a pair of columns to the lane's row, from two-word
// coordinates (planes 0 to 5).
struct SpRow2 {
    float2 xh, xl, yh, yl, th, tl;
    __device__ __forceinline__ explicit SpRow2(const float* __restrict__ r) {
        const float* q = r + (threadIdx.x & 31);
        xh = f2(q[0], q[0]); xl = f2(q[32], q[32]); yh = f2(q[64], q[64]);
        yl = f2(q[96], q[96]); th = f2(q[128], q[128]); tl = f2(q[160], q[160]);
    }
};

__device__ __forceinline__ float2 half4(const float4& v, int h) { return h ? f2(v.z, v.w) : f2(v.x, v.y); }

template <bool MASK, bool LL>
__device__ __forceinline__ void sp_add_b(float2 dx, float2 dy, float2 dt, int r0, int r1, SpRow& w) {
    const float2 r2 = fma2(dy, dy, mul2(dx, dx));
    const float2 dt2 = mul2(dt, dt);
    const float2 aB = add2(dt2, r2);
    float2 B = f2(ex2(-aB.x), ex2(-aB.y));
    if (MASK) {  // t_j != t_i
        B.x = (r0 < w.lo || r0 >= w.hi) ? B.x : 0.f;
        B.y = (r1 < w.lo || r1 >= w.hi) ? B.y : 0.f;
    }
    w.sB = add2(w.sB, B);
    if (!LL) {
        w.sBr = fma2(B, r2, w.sBr);
        w.sBt = fma2(B, dt2, w.sBt);
    }
}

// Background of `quads` x 4 buffered columns against the lane's row.
template <bool MASK, bool LL>
__device__ __forceinline__ void sp_eval_b(const SpWarp& sw, int first, int quads, SpRow& w) {
    constexpr int P = SP_BUF / 4;
    const float4* p = reinterpret_cast<const float4*>(sw.b + first);
    const SpRow2 r(sw.row);
    int4 rk = make_int4(0, 0, 0, 0);
#pragma unroll 2
    for (int q = 0; q < quads; ++q, ++p) {
        const float4 xh = p[0 * P], xl = p[1 * P], yh = p[2 * P], yl = p[3 * P], th = p[4 * P], tl = p[5 * P];
        if (MASK) rk = *reinterpret_cast<const int4*>(p + 6 * P);
#pragma unroll
        for (int h = 0; h < 2; ++h)
            sp_add_b<MASK, LL>(add2(add2(r.xh, half4(xh, h)), add2(r.xl, half4(xl, h))),
                               add2(add2(r.yh, half4(yh, h)), add2(r.yl, half4(yl, h))),
                               add2(add2(r.th, half4(th, h)), add2(r.tl, half4(tl, h))),
                               h ? rk.z : rk.x, h ? rk.w : rk.y, w);
    }
}

// Excitation of `quads` x 4 buffered columns (planes as above, then -beta, ce).
template <bool MASK, bool LL>
__device__ __forceinline__ void sp_eval_e(const SpWarp& sw, int first, int quads, float2 nomt, SpRow& w) {
    const SpRow2 r(sw.row);
#pragma unroll 1
    for (int q = 0; q < quads; ++q) {
        const float4* p = reinterpret_cast<const float4*>(sw.e + first) + q;
        const float4 xh = p[0 * SP_BUF / 4], xl = p[1 * SP_BUF / 4], yh = p[2 * SP_BUF / 4],
                     yl = p[3 * SP_BUF / 4], th = p[4 * SP_BUF / 4], tl = p[5 * SP_BUF / 4],
                     nb = p[7 * SP_BUF / 4], ce = p[8 * SP_BUF / 4];
        int4 rk;
        if (MASK) rk = *reinterpret_cast<const int4*>(p + 6 * SP_BUF / 4);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float2 dt = add2(add2(r.th, half4(th, h)), add2(r.tl, half4(tl, h)));
            const float2 dx = add2(add2(r.xh, half4(xh, h)), add2(r.xl, half4(xl, h)));
            const float2 dy = add2(add2(r.yh, half4(yh, h)), add2(r.yl, half4(yl, h)));
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

template <bool LL>
__device__ __forceinline__ void sp_background(const SpWarp& sw, int first, int quads, bool mask, SpRow& w) {
    if (mask) sp_eval_b<true, LL>(sw, first, quads, w);
    else sp_eval_b<false, LL>(sw, first, quads, w);
}

template <bool LL>
__device__ __forceinline__ void sp_excitation(const SpWarp& sw, int first, int quads, bool mask, float2 nomt, SpRow& w) {
    if (mask) sp_eval_e<true, LL>(sw, first, quads, nomt, w);
    else sp_eval_e<false, LL>(sw, first, quads, nomt, w);
}

// A listed chunk: offset of its centre from the group's, then its number, and
// SP_FAR if the sum of a first word and the offset may not be exact (above 512).
constexpr int SP_FAR = 1 << 27, SP_ID = SP_FAR - 1;

// A column's coordinates from the group's centre in two words each.
__device__ __forceinline__ void sp_two_words(const float4& a, const float4& b, const float4& off, float& xh, float& yh,
                                             float& th, float& xl, float& yl, float& tl) {
    const bool far = (__float_as_int(off.w) & SP_FAR) != 0;
    sp_shift(a.x, b.x, off.x, far, xh, xl);
    sp_shift(a.y, b.y, off.y, far, yh, yl);
    sp_shift(a.z, b.z, off.z, far, th, tl);
}

// Test the events of the n listed chunks, one per lane, for a nonzero
// background, and evaluate the survivors 32 at a time.  count: survivors so far
// (the buffer is a ring of two halves); mask: the current half holds a column
// that may share a time with a row.
template <bool LL>
__device__ __forceinline__ void sp_columns_b(const SpArgs& a, SpWarp& sw, int n, const SpGroup& gr, SpRow& w,
                                             int& count, bool& mask) {
    constexpr unsigned ALL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    const float4* ra = a.ra + lane;
    const float4* rb = a.rb + lane;
    int64_t p = static_cast<int64_t>(__float_as_int(sw.list[0].w) & SP_ID) * SP_CH;
    float4 next = ra[p], nextl = rb[p];
#pragma unroll 1
    for (int k = 0; k < n; ++k) {
        const float4 q = next, l = nextl, off = sw.list[k];
        p = static_cast<int64_t>(__float_as_int(sw.list[min(k + 1, n - 1)].w) & SP_ID) * SP_CH;
        next = ra[p];
        nextl = rb[p];
        const int id = __float_as_int(off.w);
        const uint32_t rk = __float_as_uint(q.w);
        float hx, hy, ht, lx, ly, lt;  // negated, from the group's centre
        sp_two_words(q, l, off, hx, hy, ht, lx, ly, lt);
        const float nx = hx + lx, ny = hy + ly, nt = ht + lt;
        const bool keep = sp_keep_b(gr, nx, ny, nt);  // (a padding event's time is far from any)
        const unsigned bal = __ballot_sync(ALL, keep);
        const bool any = __any_sync(ALL, keep && rk - (static_cast<uint32_t>(gr.lo_min) | SP_TIED) <
                                                     static_cast<unsigned>(gr.ties)) ||
                         (id & SP_ID) == gr.self;
        mask |= any;
        if (keep) {
            float* b = sw.b + ((count + __popc(bal & below)) & (SP_BUF - 1));
            b[0 * SP_BUF] = hx; b[1 * SP_BUF] = lx; b[2 * SP_BUF] = hy; b[3 * SP_BUF] = ly;
            b[4 * SP_BUF] = ht; b[5 * SP_BUF] = lt;
            b[6 * SP_BUF] = __int_as_float(sp_event(rk));
        }
        const int before = count;
        count += __popc(bal);
        if ((before ^ count) & 32) {
            __syncwarp();
            sp_background<LL>(sw, before & 32, 8, mask, w);
            mask = any;
            __syncwarp();
        }
    }
}

// The same for the excitation (the listed chunks from the end of the list).
template <bool LL>
__device__ __forceinline__ void sp_columns_e(const SpArgs& a, SpWarp& sw, int n, const SpGroup& gr, float omt,
                                             SpRow& w, int& count, bool& mask) {
    constexpr unsigned ALL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    const float2 nomt = f2(-omt, -omt);
    const float4* list = sw.list + SP_LIST - 1;
    int64_t p = static_cast<int64_t>(__float_as_int(list[0].w) & SP_ID) * SP_CH + lane;
    float4 na = a.ra[p], nl = a.rb[p];
    float nc = a.rc[p];
#pragma unroll 1
    for (int k = 0; k < n; ++k) {
        const float4 q = na, l = nl, off = list[-k];
        const float ce = nc;
        p = static_cast<int64_t>(__float_as_int(list[-min(k + 1, n - 1)].w) & SP_ID) * SP_CH + lane;
        na = a.ra[p];
        nl = a.rb[p];
        nc = a.rc[p];
        const int rank = sp_event(__float_as_uint(q.w));
        float hx, hy, ht, lx, ly, lt;
        sp_two_words(q, l, off, hx, hy, ht, lx, ly, lt);
        const float nx = hx + lx, ny = hy + ly, nt = ht + lt;
        const bool keep = sp_keep_e(gr, nx, ny, nt, omt, ce, l.w);
        const unsigned bal = __ballot_sync(ALL, keep);
        const bool any = __any_sync(ALL, keep && rank >= gr.lo_min);
        mask |= any;
        if (keep) {
            float* b = sw.e + ((count + __popc(bal & below)) & (SP_BUF - 1));
            b[0 * SP_BUF] = hx; b[1 * SP_BUF] = lx; b[2 * SP_BUF] = hy; b[3 * SP_BUF] = ly;
            b[4 * SP_BUF] = ht; b[5 * SP_BUF] = lt; b[6 * SP_BUF] = __int_as_float(rank);
            b[7 * SP_BUF] = l.w; b[8 * SP_BUF] = ce;
        }
        const int before = count;
        count += __popc(bal);
        if ((before ^ count) & 32) {
            __syncwarp();
            sp_excitation<LL>(sw, before & 32, 8, mask, nomt, w);
            mask = any;
            __syncwarp();
        }
    }
}

// Persistent warps over items (row group, part of the column tiles).
template <bool LL>
__global__ void __launch_bounds__(SP_THREADS, SP_BPSM) k_sweep_sp(SpArgs a, int* __restrict__ ctr, int nitems) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31;
    SpWarp& sw = reinterpret_cast<SpWarp*>(smem)[threadIdx.x >> 5];
    const double* cc = a.cc;
    chain_wait();
    if (cc[CC_VALID] == 0.0) return;
    const float omt = static_cast<float>(cc[CC_OMT]);
    const unsigned below = (1u << lane) - 1u;
    constexpr unsigned ALL = 0xffffffffu;

    for (;;) {
        int item = 0;
        if (lane == 0) item = atomicAdd(ctr + CT_WORK, 1);
        item = __shfl_sync(ALL, item, 0);
        if (item >= nitems) {
            chain_next();
            return;
        }
        const int g = item / a.parts, part = item % a.parts;
        {
            const float4 x = a.cmeta[2 * g];
            if (!(x.x <= x.y)) continue;  // padding only
        }
        SpRow w;
        SpGroup gr;
        gr.self = g;
        int e;
        {
            const int64_t p = static_cast<int64_t>(g) * SP_CH + lane;
            const float4 qa = a.ra[p], qb = a.rb[p];
            const uint32_t rk = __float_as_uint(qa.w);
            e = rk != SP_PAD ? sp_event(rk) : -1;
            float* r = sw.row + lane;
            r[0] = -sp_grid(qa.x); r[32] = -qb.x; r[64] = -sp_grid(qa.y); r[96] = -qb.y;
            r[128] = -sp_grid(qa.z); r[160] = -qb.z;
            // (as integers: the order of nonnegative floats)
            auto half = [&](float v) {
                return sp_half(__uint_as_float(__reduce_max_sync(ALL, e >= 0 ? __float_as_uint(fabsf(v)) : 0u)));
            };
            gr.hx = half(qa.x);
            gr.hy = half(qa.y);
            gr.ht = half(qa.z);
        }
        w.lo = e >= 0 ? a.lo[e] : 0;
        w.hi = e >= 0 ? a.hi[e] : 0;
        w.sB = w.sBr = w.sBt = w.sE = w.sEt = w.sEq = f2(0.f, 0.f);
        gr.lo_min = __reduce_min_sync(ALL, e >= 0 ? w.lo : 0x7fffffff);
        gr.ties = __reduce_max_sync(ALL, e >= 0 ? w.hi : 0) - gr.lo_min;
        // The lane's FP32 sums so far go to the FP64 accumulators.
        auto flush_rows = [&]() {
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
            w.sB = w.sBr = w.sBt = w.sE = w.sEt = w.sEq = f2(0.f, 0.f);
        };

        int nB = 0, nE = 0;            // columns buffered since the last flush, and where in the buffers
        bool maskB = false, maskE = false;
        int next = 0;                  // next 32 tiles (of this part) or, unsplit, 32 blocks of tiles
        int tile0 = 0;                 // current 32 tiles
        unsigned mS = 0, mT = 0;       // surviving blocks of the round, tiles of the current 32
        for (;;) {
            // list chunks that can hold a nonzero background (from the front) and
            // excitation (from the back)
            // (the rows' box and centre are read again each time: registers)
            int lB = 0, lE = 0;
            const SpBox box = sp_load(a.cmeta, g);
            const float4 ref = a.centre[g];
            while (lB + lE <= SP_LIST - 64) {
                if (mT == 0) {
                    if (a.parts == 1) {
                        const int nblk = sp_blocks(a.ntiles);
                        while (mS == 0 && next < nblk) {
                            bool nb = false, ne = false;
                            if (next + lane < nblk) sp_near(box, sp_load(a.bmeta, next + lane), omt, nb, ne);
                            mS = __ballot_sync(ALL, nb || ne);
                            next += 32;
                        }
                        if (mS == 0) break;
                        tile0 = (next - 32 + __ffs(mS) - 1) * SP_TB;
                        mS &= mS - 1;
                    } else {
                        tile0 = next;
                        if (tile0 * a.parts + part >= a.ntiles) break;
                        next += 32;
                    }
                    const int t = (tile0 + lane) * a.parts + part;
                    bool nb = false, ne = false;
                    if (t < a.ntiles) sp_near(box, sp_load(a.tmeta, t), omt, nb, ne);
                    mT = __ballot_sync(ALL, nb || ne);
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
                float4 entry = make_float4(0.f, 0.f, 0.f, 0.f);
                if (has) {
                    const SpBox q = sp_load(a.cmeta, ch);
                    sp_near(box, q, omt, nb, ne);
                    const float width = fmaxf(fmaxf(q.x1 - q.x0, q.y1 - q.y0), q.t1 - q.t0);
                    const float4 c = a.centre[ch];
                    entry = make_float4(ref.x - c.x, ref.y - c.y, ref.z - c.z, 0.f);
                    const float far = fmaxf(fmaxf(fabsf(entry.x), fabsf(entry.y)), fabsf(entry.z));
                    entry.w = __int_as_float(ch | (sp_is_far(width, far) ? SP_FAR : 0));
                }
                const unsigned kb = __ballot_sync(ALL, nb), ke = __ballot_sync(ALL, ne);
                if (nb) sw.list[lB + __popc(kb & below)] = entry;
                if (ne) sw.list[SP_LIST - 1 - lE - __popc(ke & below)] = entry;
                lB += __popc(kb);
                lE += __popc(ke);
            }
            __syncwarp();
            if (lB + lE == 0) break;
            if (lB > 0) sp_columns_b<LL>(a, sw, lB, gr, w, nB, maskB);
            if (lE > 0) sp_columns_e<LL>(a, sw, lE, gr, omt, w, nE, maskE);
            __syncwarp();
            if (nB + nE > SP_FOLD) {
                nB &= SP_BUF - 1;
                nE &= SP_BUF - 1;
                flush_rows();
            }
        }
        // what is left in the buffers, filled up to quads with columns whose
        // terms are zero
        const int hB = nB & 32, hE = nE & 32;
        nB &= 31;
        nE &= 31;
        const int qB = (nB + 3) >> 2, qE = (nE + 3) >> 2;
        if (nB + lane < 4 * qB) {
            for (int q = 0; q < SP_B_PLANES; ++q) sw.b[q * SP_BUF + hB + nB + lane] = 0.f;
            sw.b[4 * SP_BUF + hB + nB + lane] = -PAD_T;
        }
        if (nE + lane < 4 * qE) {
            for (int q = 0; q < SP_E_PLANES; ++q) sw.e[q * SP_BUF + hE + nE + lane] = 0.f;
            sw.e[8 * SP_BUF + hE + nE + lane] = -1e30f;
        }
        __syncwarp();
        sp_background<LL>(sw, hB, qB, maskB, w);
        sp_excitation<LL>(sw, hE, qE, maskE, f2(-omt, -omt), w);
        __syncwarp();
        flush_rows();
    }
}

// Queue the spatial path's staging and sweep (after k_prep has written the
// per-call constants and zeroed the accumulators).  The records take the place
// of the staged records of the other paths.
cudaError_t spatial_launch(hawkes_ctx* c, int model1, int llonly) {
    SpatialState* sp = c->sp;
    SpArgs a;
    float4* ra = reinterpret_cast<float4*>(c->rec);
    float4* rb = ra + c->npad;
    float* rc = reinterpret_cast<float*>(rb + c->npad);
    float4* cmeta = sp->meta;
    float4* tmeta = cmeta + 16 * static_cast<size_t>(sp->ntiles);
    float4* bmeta = tmeta + 2 * static_cast<size_t>(sp->ntiles);
    const int nblk = sp_blocks(sp->ntiles);
    float4* centre = bmeta + 2 * static_cast<size_t>(nblk);
    cudaError_t err = launch_chained(k_sp_prep, std::min(sp->ntiles, 8 * c->sms), TC, 0, c->stream, eval_desc(c),
                                     sp->rank, model1, ra, rb, rc, cmeta, tmeta, centre, sp->ntiles);
    if (err != cudaSuccess) return err;
    a.ra = ra; a.rb = rb; a.rc = rc; a.lo = c->lo; a.hi = c->hi; a.cc = c->cc; a.acc = c->acc;
    a.cmeta = cmeta; a.tmeta = tmeta; a.bmeta = bmeta; a.centre = centre;
    a.npad = c->npad;
    a.ntiles = sp->ntiles;
    a.groups = static_cast<int>((c->n + SP_CH - 1) / SP_CH);
    // Few rows: several warps share a group's columns, until there are a
    // resident CTA's worth of warps for every SM.
    const size_t smem = SP_WARPS * sizeof(SpWarp);
    auto* kern = llonly ? k_sweep_sp<true> : k_sweep_sp<false>;
    a.parts = 1;
    while (a.parts < 64 && 2 * a.parts <= a.ntiles &&
           static_cast<int64_t>(a.groups) * a.parts < static_cast<int64_t>(c->sms) * SP_BPSM * SP_WARPS)
        a.parts *= 2;
    if (a.parts == 1) {
        err = launch_chained(k_sp_blocks, nblk, SP_TB, 0, c->stream, tmeta, bmeta, sp->ntiles, c->cc);
        if (err != cudaSuccess) return err;
    }
    const int64_t nitems = static_cast<int64_t>(a.groups) * a.parts;
    const int grid = static_cast<int>(std::min<int64_t>((nitems + SP_WARPS - 1) / SP_WARPS,
                                                        static_cast<int64_t>(c->sms) * SP_BPSM));
    return launch_chained(kern, grid, SP_THREADS, smem, c->stream, a, c->ctr, static_cast<int>(nitems));
}

cudaError_t spatial_setup_attributes() {
    for (auto* k : {k_sweep_sp<false>, k_sweep_sp<true>}) {
        const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   static_cast<int>(SP_WARPS * sizeof(SpWarp)));
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace hk

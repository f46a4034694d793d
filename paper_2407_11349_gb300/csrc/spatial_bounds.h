// The tests of the spatial skip (sweep_spatial.cu): which columns can hold a
// nonzero term for a group of rows, and the coordinates they are formed from.
// Plain C++ for the device and the host, so that they can be checked without a
// GPU.
#pragma once

#include <math.h>
#include <stdint.h>

#include "spatial_order.h"

namespace hk {

// The point tests allow for the rounding of the points: 2^-24 of their distance
// from the reference point, and of half a chunk's width.
constexpr float SP_EPS = 4.76837158203125e-07f;
constexpr float SP_OUT = 1.f + 9.5367431640625e-07f, SP_IN = 1.f - 9.5367431640625e-07f;
constexpr float SP_ZERO = 128.f;       // exponent beyond which a term counts as zero (126 + margin)

// Bounds of a set of events, in scaled units: box, time range, largest ce,
// smallest beta.  Empty: x0 > x1.
struct SpBox {
    float x0, x1, y0, y1, t0, t1, ce, beta;
};

SP_HD SpBox sp_empty() {
    return SpBox{1e30f, -1e30f, 1e30f, -1e30f, 1e30f, -1e30f, -1e30f, 1e30f};
}
SP_HD void sp_join(SpBox& a, const SpBox& b) {
    a.x0 = fminf(a.x0, b.x0); a.x1 = fmaxf(a.x1, b.x1);
    a.y0 = fminf(a.y0, b.y0); a.y1 = fmaxf(a.y1, b.y1);
    a.t0 = fminf(a.t0, b.t0); a.t1 = fmaxf(a.t1, b.t1);
    a.ce = fmaxf(a.ce, b.ce); a.beta = fminf(a.beta, b.beta);
}
// Widen [lo, hi] by 2^-22 of its magnitude: more than the rounding to FP32 of
// its own ends and of any point compared with it nearby.
SP_HD void sp_widen(float& lo, float& hi) {
    const float s = 2.384185791015625e-07f * fmaxf(fabsf(lo), fabsf(hi));
    lo -= s;
    hi += s;
}

// Middle of a range on a grid of 1/16, so that differences of neighbouring
// chunks' centres are exact in FP32 (beyond 2^20 FP32's own grid is coarser).
SP_HD float sp_mid(float a, float b) {
    const float m = 0.5f * a + 0.5f * b;
    return fabsf(m) < 1048576.f ? rintf(m * 16.f) * 0.0625f : m;
}

// hi + lo = a + d exactly, lo0 added to lo.
SP_HD void sp_two_sum(float a, float d, float lo0, float& hi, float& lo) {
    hi = a + d;
    const float z = hi - a;
    lo = ((a - (hi - z)) + (d - z)) + lo0;
}

// First word of a two-word coordinate: on a grid of 2^-14 for |a| < 256, so that
// first words' differences are exact.  (FP32 has steps of 2^-14 from 512 to 1,024.)
SP_HD float sp_grid(float a) { return (a + 768.f) - 768.f; }

// c - (xh + xl), and what sp_grid leaves of it.  (In FP32: FP64 arithmetic is what
// staging waits for.)
SP_HD void sp_recentre(float c, float xh, float xl, float& hi, float& lo) {
    float h, l;
    sp_two_sum(-xh, c, -xl, h, l);
    sp_two_sum(h, l, 0.f, hi, lo);
    lo += hi - sp_grid(hi);
}

// Can a column of box (or point) c hold a nonzero background / excitation term
// for some row of box w?
SP_HD float sp_gap(float lo, float hi, float a0, float a1) {
    return fmaxf(0.f, fmaxf(a0 - hi, lo - a1));
}
SP_HD void sp_near(const SpBox& w, const SpBox& c, float omt, bool& nb, bool& ne) {
    const float dx = sp_gap(w.x0, w.x1, c.x0, c.x1), dy = sp_gap(w.y0, w.y1, c.y0, c.y1);
    const float r2 = fmaf(dx, dx, dy * dy), g = sp_gap(w.t0, w.t1, c.t0, c.t1);
    nb = !(fmaf(g, g, r2) > SP_ZERO);  // (negated: a NaN is kept, and reported as ever)
    ne = c.t0 <= w.t1 && !(c.ce - omt * fmaxf(0.f, w.t0 - c.t1) - c.beta * r2 < -SP_ZERO);
}

// A row group as the column tests see it: half widths of its rows about its
// centre, and the range of time-order indices that some row must be compared
// with one by one (ties; the excitation's first later event).
struct SpGroup {
    float hx, hy, ht;
    int lo_min, ties;  // [lo_min, lo_min + ties)
    int self;          // its own chunk
};

// Half width of rows whose largest distance from the centre is v, not below the
// true one.
SP_HD float sp_half(float v) { return v * SP_OUT + SP_EPS; }
// Distance beyond the group's half width, not above the true one.
SP_HD float sp_beyond(float d, float half) { return fmaxf(0.f, fmaf(fabsf(d), SP_IN, -half)); }

// Can a column at (x, y, t) from the group's centre (negated: t > 0 is earlier)
// hold a nonzero background / excitation term for some row of the group?
// (Negated comparisons: a NaN is kept.)
SP_HD bool sp_keep_b(const SpGroup& gr, float x, float y, float t) {
    const float dx = sp_beyond(x, gr.hx), dy = sp_beyond(y, gr.hy), dt = sp_beyond(t, gr.ht);
    return !(fmaf(dt, dt, fmaf(dx, dx, dy * dy)) > SP_ZERO);
}
SP_HD bool sp_keep_e(const SpGroup& gr, float x, float y, float t, float omt, float ce, float neg_beta) {
    const float dx = sp_beyond(x, gr.hx), dy = sp_beyond(y, gr.hy);
    const float gap = fmaxf(0.f, fmaf(t, SP_IN, -gr.ht));
    return -t <= gr.ht + fabsf(t) * SP_EPS && !(ce - omt * gap + neg_beta * fmaf(dx, dx, dy * dy) < -SP_ZERO);
}

// May the sum of a first word and the offset between two centres be inexact
// (above 512)?  width: of the column's chunk.
SP_HD bool sp_is_far(float width, float offset) { return !(width + offset <= 256.f); }

// A column's coordinate from the group's centre in two words: (a, b) from its own
// chunk's centre, off the offset between the centres.
SP_HD void sp_shift(float a, float b, float off, bool far, float& hi, float& lo) {
    if (far) {
        sp_two_sum(sp_grid(a), off, b, hi, lo);
    } else {
        hi = sp_grid(a) + off;
        lo = b;
    }
}

}  // namespace hk

"""What the spatial skip leaves out is an exact FP32 zero: the library's own order
and tests (csrc/spatial_order.h, csrc/spatial_bounds.h) compiled and run on the
host, against every pair's exponents in FP64.

As the kernels do: events in the k-d order, records from their chunk's centre in
two FP32 words, boxes of chunks, tiles and blocks of tiles; a chunk is listed for
a group of 32 rows by boxes, and its events are tested one by one.  Checked for
every pair of rows and columns:
  - left out of the background: the base-2 exponent dt~^2 + r~^2 is above 126, or
    the events share their time;
  - left out of the excitation: the exponent ce - omega~ dt~ - beta r~^2 is below
    -126, or the source is not earlier;
  - a listed chunk's tile and block of tiles pass the same test."""
import ctypes
import os
import subprocess
import textwrap

import numpy as np
import pytest

from paper_2407_11349_gb300 import synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2407_11349_gb300", "csrc")

SRC = textwrap.dedent("""
    #include <algorithm>
    #include <cmath>
    #include <vector>
    #include "spatial_bounds.h"
    using namespace hk;
    struct Word { float h, l; };
    // out: pairs kept (background, excitation), pairs left out, violations of
    // the background, the excitation, the hierarchy
    extern "C" void check(int n, const double* t, const double* x, const double* y, const double* s,
                          const int* county, int n_counties, const double* p, const double* q, long window, long* out) {
        const double tx = p[1], tt = p[2], om = p[4], h = p[5], L = std::log2(std::exp(1.0));
        const double ax = L / (2 * tx * tx), at = L / (2 * tt * tt), kx = std::sqrt(ax), kt = std::sqrt(at);
        const float omt = float(om * L / kt);
        const double beta0 = tx * tx / (h * h);
        std::vector<double> vt(t, t + n), vx(x, x + n), vy(y, y + n);
        std::vector<int32_t> vc(county, county + n);
        std::vector<SpPoint> pt = sp_points(vt, vx, vy, vc, n_counties, q[0], q[1]);
        sp_split_windows(pt, window);
        const int nch = (n + SP_CH - 1) / SP_CH, per = SP_TILE / SP_CH;
        std::vector<Word> X(n), Y(n), T(n);
        std::vector<float> ce(n), nbeta(n);
        std::vector<SpBox> box(nch, sp_empty());
        std::vector<float> cx(nch), cy(nch), ct(nch);
        for (int c = 0; c < nch; ++c) {
            const int a = c * SP_CH, b = std::min(n, a + SP_CH);
            std::vector<Word> wx(b - a), wy(b - a), wt(b - a);
            for (int k = a; k < b; ++k) {
                const int e = pt[k].e;
                auto two = [](double v) { const float f = float(v); return Word{f, float(v - double(f))}; };
                wx[k - a] = two(x[e] * kx); wy[k - a] = two(y[e] * kx); wt[k - a] = two((t[e] - t[0]) * kt);
                ce[k] = float(-2.0 * std::log2(s[e]));
                nbeta[k] = -float(beta0 / (s[e] * s[e]));
                const float fx = wx[k - a].h, fy = wy[k - a].h, ft = wt[k - a].h;
                sp_join(box[c], SpBox{fx, fx, fy, fy, ft, ft, ce[k], -nbeta[k]});
            }
            cx[c] = sp_mid(box[c].x0, box[c].x1); cy[c] = sp_mid(box[c].y0, box[c].y1); ct[c] = sp_mid(box[c].t0, box[c].t1);
            for (int k = a; k < b; ++k) {
                sp_recentre(cx[c], wx[k - a].h, wx[k - a].l, X[k].h, X[k].l);
                sp_recentre(cy[c], wy[k - a].h, wy[k - a].l, Y[k].h, Y[k].l);
                sp_recentre(ct[c], wt[k - a].h, wt[k - a].l, T[k].h, T[k].l);
            }
            sp_widen(box[c].x0, box[c].x1); sp_widen(box[c].y0, box[c].y1); sp_widen(box[c].t0, box[c].t1);
        }
        const int ntile = (nch + per - 1) / per, nblk = (ntile + 31) / 32;
        std::vector<SpBox> tile(ntile, sp_empty()), blk(nblk, sp_empty());
        for (int c = 0; c < nch; ++c) { sp_join(tile[c / per], box[c]); sp_join(blk[c / per / 32], box[c]); }
        for (int g = 0; g < nch; ++g) {
            const int ra = g * SP_CH, rb = std::min(n, ra + SP_CH);
            SpGroup gr{};
            for (int k = ra; k < rb; ++k) {
                gr.hx = std::max(gr.hx, std::fabs(X[k].h)); gr.hy = std::max(gr.hy, std::fabs(Y[k].h));
                gr.ht = std::max(gr.ht, std::fabs(T[k].h));
            }
            gr.hx = sp_half(gr.hx); gr.hy = sp_half(gr.hy); gr.ht = sp_half(gr.ht);
            for (int c = 0; c < nch; ++c) {
                bool nb, ne, tb, te, bb, be;
                sp_near(box[g], box[c], omt, nb, ne);
                sp_near(box[g], tile[c / per], omt, tb, te);
                sp_near(box[g], blk[c / per / 32], omt, bb, be);
                if ((nb || ne) && !((tb || te) && (bb || be))) ++out[5];
                const SpBox& w = box[c];
                const float width = std::max(std::max(w.x1 - w.x0, w.y1 - w.y0), w.t1 - w.t0);
                const float ox = cx[g] - cx[c], oy = cy[g] - cy[c], ot = ct[g] - ct[c];
                const bool far = sp_is_far(width, std::max(std::max(std::fabs(ox), std::fabs(oy)), std::fabs(ot)));
                for (int k = c * SP_CH; k < std::min(n, c * SP_CH + SP_CH); ++k) {
                    Word a, b, d;
                    sp_shift(X[k].h, X[k].l, ox, far, a.h, a.l);
                    sp_shift(Y[k].h, Y[k].l, oy, far, b.h, b.l);
                    sp_shift(T[k].h, T[k].l, ot, far, d.h, d.l);
                    const float fx = a.h + a.l, fy = b.h + b.l, ft = d.h + d.l;
                    const bool kb = nb && sp_keep_b(gr, fx, fy, ft);
                    const bool ke = ne && sp_keep_e(gr, fx, fy, ft, omt, ce[k], nbeta[k]);
                    const int j = pt[k].e;
                    for (int r = ra; r < rb; ++r) {
                        const int i = pt[r].e;
                        const double dt = t[i] - t[j], dx = x[i] - x[j], dy = y[i] - y[j], r2 = dx * dx + dy * dy;
                        if (!kb && dt != 0 && !(dt * dt * at + r2 * ax > 126.0)) ++out[3];
                        if (!ke && dt > 0 &&
                            !(-2 * std::log2(s[j]) - om * L * dt - r2 * L / (2 * h * h * s[j] * s[j]) < -126.0)) ++out[4];
                    }
                    const long rows = rb - ra;
                    out[0] += kb ? rows : 0; out[1] += ke ? rows : 0; out[2] += !kb && !ke ? rows : 0;
                }
            }
        }
    }
    """)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("spatial")
    with open(d / "t.cpp", "w") as f:
        f.write(SRC)
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-pthread", "-I", CSRC, str(d / "t.cpp"), "-o",
                    str(d / "t.so")], check=True)
    return ctypes.CDLL(str(d / "t.so"))


def run(lib, t, x, y, s, county, n_counties, p, order, window):
    D, I = ctypes.POINTER(ctypes.c_double), ctypes.POINTER(ctypes.c_int)
    arr = [np.ascontiguousarray(v, dtype=np.float64) for v in (t, x, y, s, p, order)]
    c = np.ascontiguousarray(county, dtype=np.int32)
    out = (ctypes.c_long * 6)()
    ptr = [v.ctypes.data_as(D) for v in arr]
    lib.check(len(t), *ptr[:4], c.ctypes.data_as(I), n_counties, ptr[4], ptr[5], ctypes.c_long(window), out)
    kb, ke, skipped, *wrong = list(out)
    assert wrong == [0, 0, 0], wrong
    return kb, ke, skipped


P0 = synth.DEFAULT_PARAMS


@pytest.mark.parametrize("seed,window,p", [(1, 512, P0), (2, 1024, (2.0, 50.0, 10.0, 0.9, 0.05, 20.0)),
                                           (3, 256, (0.5, 5.0, 2.0, 0.3, 1.5, 0.5)), (4, 131072, P0)])
def test_regular_maps_ties_and_windows(lib, seed, window, p):
    ds = synth.grid_dataset(3001, 1200.0, 20, 20, seed=seed)
    if seed == 1:
        ds = synth.integer_day_times(ds)
    # ordered with and without counties, and by another call's bandwidths
    for cty, order in ((0, p[1:3]), (ds.counties.n, p[1:3]), (0, (0.01 * p[1], 100.0 * p[2]))):
        _, _, skipped = run(lib, ds.t, ds.x, ds.y, ds.s, ds.county, cty, p, order, window)
        assert skipped > 0.2 * ds.n ** 2  # the check is exercised


@pytest.mark.parametrize("shift", [0.0, 5.0e4, -5.0e6])
@pytest.mark.parametrize("spread", [3.0, 3000.0])
def test_clusters_and_centres_beyond_the_exact_grid(lib, spread, shift):
    rng = np.random.default_rng(int(spread))
    n = 2500
    x, y, t = rng.uniform(0, spread, n), rng.uniform(0, spread, n), rng.uniform(0.1, 1000.0, n)
    for k in range(3):
        m = slice(400 * k, 400 * k + 400)
        x[m], y[m] = 0.2 * spread * (k + 0.5) + rng.normal(0, 5.0, 400), 0.5 * spread + rng.normal(0, 5.0, 400)
        t[m] = 200.0 * (k + 1) + rng.uniform(0, 5.0, 400)
    o = np.argsort(t)
    county = np.arange(n) % 7
    s = rng.uniform(0.2, 4.0, 7)[county]
    for p in (P0, (0.5, 0.02, 7.0, 0.3, 0.2, 0.002), (0.5, 80.0, 60.0, 0.3, 0.02, 20.0)):
        run(lib, t[o], x[o] + shift, y[o] - shift, s, county, 0, p, p[1:3], 131072)

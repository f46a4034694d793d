// The order of the events for the spatial skip (sweep_spatial.cu), on the host:
// time windows, each split by a k-d tree down to chunks of SP_CH events.  Plain
// C++, so that it can be compiled and checked without a GPU.
#pragma once

#include <stdint.h>

#include <algorithm>
#include <exception>
#include <thread>
#include <vector>

namespace hk {

constexpr int SP_CH = 32;     // events per chunk: a row group, and the finest column unit
constexpr int SP_TILE = 256;  // events per tile

// A position's entry in the order: the event's index in time order, and whether
// other events share its time; SP_PAD for padding.  (Indices end below 2^31 - 4,096,
// hawkes_set_events, so no event's entry is SP_PAD.)
#ifdef __CUDACC__
#define SP_HD __host__ __device__ __forceinline__
#else
#define SP_HD inline
#endif
constexpr uint32_t SP_TIED = 1u << 31, SP_PAD = ~0u;
SP_HD uint32_t sp_rank(int32_t e, bool tied) { return static_cast<uint32_t>(e) | (tied ? SP_TIED : 0u); }
SP_HD int32_t sp_event(uint32_t rank) { return static_cast<int32_t>(rank & ~SP_TIED); }

struct SpPoint {
    float c[3];
    int32_t e;
};

// A point's coordinate: finite, so that the points can be ordered.  (Sums and
// differences of coordinates near the end of the FP64 range are not.)
inline float sp_coord(double v) {
    return v != v ? 0.f : static_cast<float>(std::min(std::max(v, -1e30), 1e30));
}

// The events as points of the tree.  Locations that will be redrawn inside their
// counties (n_counties > 0) enter as the county's mean plus a fifth of the offset
// from it.  x and y are overwritten.
inline std::vector<SpPoint> sp_points(const std::vector<double>& t, std::vector<double>& x, std::vector<double>& y,
                                      const std::vector<int32_t>& county, int32_t n_counties, double tau_x,
                                      double tau_t) {
    const size_t n = t.size();
    if (n_counties > 0) {
        std::vector<double> mx(n_counties, 0.0), my(n_counties, 0.0), cnt(n_counties, 0.0);
        for (size_t i = 0; i < n; ++i) {
            mx[county[i]] += x[i];
            my[county[i]] += y[i];
            cnt[county[i]] += 1.0;
        }
        for (size_t i = 0; i < n; ++i) {
            const double cx = mx[county[i]] / cnt[county[i]], cy = my[county[i]] / cnt[county[i]];
            x[i] = cx + 0.2 * (x[i] - cx);
            y[i] = cy + 0.2 * (y[i] - cy);
        }
    }
    std::vector<SpPoint> pt(n);
    for (size_t i = 0; i < n; ++i)
        pt[i] = SpPoint{{sp_coord((x[i] - x[0]) / tau_x), sp_coord((y[i] - y[0]) / tau_x),
                         sp_coord((t[i] - t[0]) / tau_t)},
                        static_cast<int32_t>(i)};
    return pt;
}

// Split [a, b) at medians of its widest side, down to chunks; parts stay whole
// tiles while larger than a tile.
inline void sp_split(SpPoint* a, SpPoint* b) {
    while (b - a > SP_CH) {
        const int64_t len = b - a, unit = len > SP_TILE ? SP_TILE : SP_CH;
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

// Split every time window (whole tiles) of about `window` points, on a few host
// threads for many points.
inline void sp_split_windows(std::vector<SpPoint>& pt, int64_t window) {
    const int64_t n = static_cast<int64_t>(pt.size());
    const int64_t w = (window + SP_TILE - 1) / SP_TILE * SP_TILE;
    const int64_t nw = (n + w - 1) / w;
    auto work = [&](int64_t k0, int64_t step) {
        for (int64_t k = k0; k < nw; k += step) sp_split(pt.data() + k * w, pt.data() + std::min(n, (k + 1) * w));
    };
    const int64_t nth = std::min<int64_t>(nw, n > 50000 ? 8 : 1);
    std::vector<std::thread> th;
    th.reserve(static_cast<size_t>(nth));  // (may throw: no thread runs yet)
    int64_t started = 1;  // this thread takes window 0, nth, 2 nth, ...
    try {
        for (; started < nth; ++started) th.emplace_back(work, started, nth);
    } catch (const std::exception&) {  // no more threads, or no memory for one: the rest runs here
    }
    work(0, nth);
    for (int64_t k = started; k < nth; ++k) work(k, nth);
    for (std::thread& q : th) q.join();
}

}  // namespace hk

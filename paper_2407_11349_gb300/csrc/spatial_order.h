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

struct SpPoint {
    float c[3];
    int32_t e;
};

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

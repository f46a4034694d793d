"""The event order of the spatial skip (csrc/spatial_order.h), compiled and run
on the host without a GPU."""
import os
import subprocess
import textwrap

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2407_11349_gb300", "csrc")


def run_cpp(tmp_path, src, *args):
    cpp, exe = str(tmp_path / "t.cpp"), str(tmp_path / "t")
    with open(cpp, "w") as f:
        f.write(textwrap.dedent(src))
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, cpp, "-o", exe], check=True)
    return subprocess.run([exe, *map(str, args)], capture_output=True, text=True, timeout=300)


@pytest.mark.parametrize("fail_at", range(12))
def test_out_of_memory_while_threads_run(tmp_path, fail_at):
    """The fail_at-th allocation of the split throws: the caller sees bad_alloc
    or the whole order, and the process does not end."""
    r = run_cpp(tmp_path, """
        #include <cstdio>
        #include <cstdlib>
        #include <new>
        #include "spatial_order.h"
        static long left = -1;
        void* operator new(size_t n) {
            if (left >= 0 && left-- == 0) throw std::bad_alloc();
            if (void* p = std::malloc(n)) return p;
            throw std::bad_alloc();
        }
        void operator delete(void* p) noexcept { std::free(p); }
        void operator delete(void* p, size_t) noexcept { std::free(p); }
        int main(int, char** argv) {
            const int n = 60000;
            std::vector<hk::SpPoint> pt(n);
            for (int i = 0; i < n; ++i) pt[i] = {{float(i * 7919 % n), float(i * 104729 % n), float(i)}, i};
            left = std::atol(argv[1]);
            try {
                hk::sp_split_windows(pt, 4096);
            } catch (const std::bad_alloc&) {
                std::puts("bad_alloc");
                return 0;
            }
            left = -1;
            std::vector<char> seen(n, 0);
            for (const auto& p : pt) seen[p.e] = 1;
            for (char s : seen) if (!s) return 1;
            std::puts("ordered");
        }
        """, fail_at)
    assert r.returncode == 0 and r.stdout.strip() in ("bad_alloc", "ordered"), (r.returncode, r.stdout, r.stderr)


@pytest.mark.parametrize("size", [1e3, 1.7e308])
def test_order_is_a_permutation_at_any_finite_coordinate(tmp_path, size):
    """County means, and differences, of finite coordinates may overflow; the
    points keep an order all the same (a NaN would leave none, and the split could
    then run outside its range)."""
    r = run_cpp(tmp_path, """
        #include <cmath>
        #include <cstdio>
        #include <cstdlib>
        #include "spatial_order.h"
        int main(int, char** argv) {
            const int n = 5000;
            const double size = std::atof(argv[1]);
            std::vector<double> t(n), x(n), y(n);
            std::vector<int32_t> county(n);
            for (int i = 0; i < n; ++i) {
                t[i] = 1.0 + i / 3;
                x[i] = size * (((i * 7919) % 1000) / 500.0 - 1.0);
                y[i] = (i % 5 ? size : -size) * 0.9;
                county[i] = i % 7;
            }
            std::vector<hk::SpPoint> pt = hk::sp_points(t, x, y, county, 7, 1.0, 1.0);
            for (const auto& p : pt)
                for (float c : p.c)
                    if (!std::isfinite(c)) return 2;
            hk::sp_split_windows(pt, 1024);
            std::vector<char> seen(n, 0);
            for (const auto& p : pt) seen[p.e] = 1;
            for (char s : seen) if (!s) return 1;
        }
        """, repr(size))
    assert r.returncode == 0, r.returncode


def test_every_event_index_has_an_entry(tmp_path):
    """Indices up to the largest that hawkes_set_events accepts (n at most
    2^31 - 4,096), tied or not, come back whole and are never the padding."""
    r = run_cpp(tmp_path, """
        #include "spatial_order.h"
        int main() {
            const int64_t last = (int64_t(1) << 31) - 4097;
            for (int64_t e : {int64_t(0), int64_t(1), (int64_t(1) << 30) - 1, int64_t(1) << 30, last})
                for (bool tied : {false, true}) {
                    const uint32_t r = hk::sp_rank(int32_t(e), tied);
                    if (hk::sp_event(r) != e || r == hk::SP_PAD || bool(r & hk::SP_TIED) != tied) return 1;
                }
        }
        """)
    assert r.returncode == 0

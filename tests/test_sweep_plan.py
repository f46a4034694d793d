"""The plan of the pair sweep (csrc/sweep_plan.h), compiled and run on the host
without a GPU."""
import os
import subprocess
import textwrap

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2407_11349_gb300", "csrc")


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    """plan(sms, band, n, ...): (column split, items' column tiles, band,
    allocations made), for the default variant's row tiles."""
    d = tmp_path_factory.mktemp("plan")
    with open(d / "t.cpp", "w") as f:
        f.write(textwrap.dedent("""
            #include <cstdio>
            #include <cstdlib>
            #include <new>
            #include "sweep_plan.h"
            static long news = 0;
            void* operator new(size_t n) { ++news; return std::malloc(n); }
            void operator delete(void* p) noexcept { std::free(p); }
            void operator delete(void* p, size_t) noexcept { std::free(p); }
            int main(int argc, char** argv) {
                static int64_t ns[64];
                for (int k = 3; k < argc; ++k) ns[k - 3] = std::atoll(argv[k]);
                const long before = news;
                const hk::SweepPlan pl = hk::sweep_plan(ns, argc - 3, std::atoi(argv[1]), hk::PlanKernels{2048, 1, 128}, 0,
                                                        std::atoi(argv[2]) != 0);
                std::printf("%d %d %d %ld", int(pl.split), pl.chunk, int(pl.band), news - before);
            }
            """))
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, str(d / "t.cpp"), "-o", str(d / "t")], check=True)

    def run(sms, band, *ns):
        r = subprocess.run([str(d / "t"), str(sms), str(int(band)), *map(str, ns)], capture_output=True, text=True, check=True)
        return tuple(int(v) for v in r.stdout.split())

    return run


def test_planning_allocates_nothing(plan):
    for band in (False, True):
        for ns in ((1,), (2000,), (65_536,), (1_000_000,), (5000, 20_000, 300)):
            assert plan(152, band, *ns)[3] == 0


# Sweep times of both plans measured on 152 SMs (ms; space-time background, 1,200
# days): events, column split alone, row tiles with the band
MEASURED = [(4000, 0.0189, 0.0734), (6000, 0.0347, 0.0734), (8000, 0.0504, 0.0735), (9000, 0.0551, 0.0732),
            (9750, 0.0590, 0.0735), (10_250, 0.0635, 0.0746), (11_000, 0.0685, 0.0752), (11_200, 0.0752, 0.0763),
            (11_500, 0.0757, 0.0762), (12_000, 0.0762, 0.0772), (12_250, 0.0767, 0.0799), (13_000, 0.0943, 0.1301),
            (14_500, 0.1124, 0.1300), (15_500, 0.1241, 0.1303), (16_450, 0.1292, 0.1373), (16_800, 0.1394, 0.1382),
            (17_103, 0.1432, 0.1376), (17_500, 0.1436, 0.1812), (18_250, 0.1627, 0.1878), (18_500, 0.1688, 0.1899),
            (20_000, 0.1901, 0.2013), (20_800, 0.2033, 0.2265), (21_200, 0.2115, 0.2264), (21_600, 0.2131, 0.2439),
            (22_000, 0.2263, 0.2428), (23_250, 0.2484, 0.2481), (23_700, 0.2616, 0.2475), (24_100, 0.2653, 0.2478),
            (24_550, 0.2751, 0.2477), (25_000, 0.2868, 0.2969), (26_000, 0.3108, 0.3231), (27_000, 0.3287, 0.3371),
            (27_200, 0.3330, 0.3389), (27_600, 0.3422, 0.3383), (28_500, 0.3628, 0.3532), (30_000, 0.4010, 0.3779),
            (31_500, 0.4424, 0.4216), (33_000, 0.4779, 0.4811), (34_500, 0.5229, 0.4807), (36_000, 0.5692, 0.5632),
            (37_000, 0.6011, 0.5993), (40_000, 0.6954, 0.6710), (43_000, 0.8008, 0.7217), (48_000, 0.9915, 0.9226),
            (53_000, 1.2090, 1.0914), (58_000, 1.4430, 1.3138), (65_536, 1.8294, 1.6654)]


@pytest.mark.parametrize("n,split_ms,band_ms", MEASURED)
def test_the_chosen_plan_is_within_3_percent_of_the_faster_one(plan, n, split_ms, band_ms):
    split, _, band, _ = plan(152, True, n)
    assert bool(split) != bool(band)
    assert (split_ms if split else band_ms) <= 1.03 * min(split_ms, band_ms)


def test_ranges(plan):
    """Small sums have no columns below their row tile; from 28,000 events on,
    alone or together in a batch, the row tiles are taken; and in between the
    plan changes where the comment of the rule says it can."""
    assert all(plan(152, True, n)[:1] == (1,) for n in (1, 300, 2000, 2048))
    assert all(plan(152, True, n)[2] == 1 for n in range(28_000, 120_000, 1_777))
    assert plan(152, True, 20_000, 20_000)[2] == 1
    assert all(plan(152, False, n)[2] == 0 for n in (2000, 20_000, 65_536))  # no band for the allocation-free call

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

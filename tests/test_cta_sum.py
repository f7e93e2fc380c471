"""first_warp_sum (csrc/evx_cta_sum.cuh) run on the CPU: one thread per lane, a shuffle
that meets at a barrier and refuses masks naming lanes that the CTA does not have. The
z passes call it with 18 to 30 threads on short grids (20^3: 20)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2507_21748_gb300", "csrc")

PROGRAM = r"""
#include <barrier>
#include <cmath>
#include <cstdio>
#include <memory>
#include <thread>
#include <vector>
#define __device__
#define __forceinline__ inline
static int g_live;
static bool g_bad;
static double g_val[32];
static std::unique_ptr<std::barrier<>> g_bar;
static thread_local int t_lane;
static double __shfl_down_sync(unsigned mask, double v, int o) {
    const unsigned exist = g_live == 32 ? 0xffffffffu : (1u << g_live) - 1u;
    if (mask != exist) g_bad = true;  // a lane that is not there, or one left out
    g_val[t_lane] = v;
    g_bar->arrive_and_wait();
    const int src = t_lane + o;
    const double r = src > 31 ? v : src >= g_live ? NAN : g_val[src];
    g_bar->arrive_and_wait();
    return r;
}
#include "evx_cta_sum.cuh"
int main() {
    for (int n = 1; n <= 256; ++n) {
        std::vector<double> red(n);
        double want = 0.0;
        for (int i = 0; i < n; ++i) want += red[i] = 1.0 + i * i;  // whole numbers: any order is exact
        g_live = n < 32 ? n : 32;
        g_bad = false;
        g_bar = std::make_unique<std::barrier<>>(g_live);
        double got = NAN;
        std::vector<std::thread> ts;
        for (int l = 0; l < g_live; ++l)
            ts.emplace_back([&, l] {
                t_lane = l;
                const double s = evx::first_warp_sum(red.data(), n, l);
                if (l == 0) got = s;
            });
        for (auto& t : ts) t.join();
        if (g_bad || got != want) {
            std::printf("n = %d: %s, sum %g, expected %g\n", n, g_bad ? "bad mask" : "masks fine", got, want);
            return 1;
        }
    }
    return 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_first_warp_sum_uses_existing_lanes_only(tmp_path):
    src, exe = tmp_path / "cta_sum.cpp", tmp_path / "cta_sum"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++20", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout


def test_z_passes_end_their_sums_with_it():
    for name in ("evx_mixed_z.cu", "evx_staged.cu"):
        with open(os.path.join(CSRC, name)) as f:
            text = f.read()
        assert text.count("first_warp_sum(red, nthr, tid)") == 2 and "__shfl" not in text, name

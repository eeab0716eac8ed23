"""The launch plan (csrc/pt_host.h, compiled for the host) against the search that it shortens: every shape
estimated in full, and a batch's instances one by one."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_1605_03607_gb300", "csrc")

DRIVER = r"""
#include <cstdio>
#include <random>
#include "pt_host.h"
using namespace ptg;
static const int WS[] = {1, 2, 3, 4, 6, 8, 12, 16, 24, 32};
static int units_of(int L) { return (L & 1) ? L * L / 2 + 1 : (L / 2) * (L / 2); }
static LaneShape full_plan(int L, int NT, int kt, int R, int n_inst, bool walk, int sms, int cap)
{
    LaneShape best;
    double best_t = 1e300;
    for (int gr = 1; gr <= 8 && gr <= R; ++gr)
        for (int G = 1; G <= LANE_GROUPS && (G - 1) * gr < R; ++G)
            for (int span = 0; span < 2; ++span) {
                const int64_t per = (R + gr - 1) / gr;
                if (span && (n_inst == 1 || per % G == 0)) continue;
                const int64_t smem = lane_layout(L, NT, kt, gr, G, walk, span ? 2 : 1).bytes;
                if (smem > cap) continue;
                for (int W : WS) {
                    LaneShape s;
                    s.W = W; s.gr = gr; s.G = G; s.span = span != 0;
                    const int threads = lane_threads(NT, s);
                    if (threads > LANE_THREADS || (W > units_of(L) && W > 1)) break;
                    const int fit = lane_counted(threads, smem);
                    const int64_t ctas = span ? (n_inst * per + G - 1) / G : n_inst * ((per + G - 1) / G), wave = (int64_t)fit * sms;
                    const int rest = (int)((ctas % wave + sms - 1) / sms);
                    const double t = (double)(ctas / wave) * lane_clocks(L, NT, s, fit) + (rest ? lane_clocks(L, NT, s, rest) : 0.0);
                    if (t < best_t * 0.999) { best_t = t; best = s; }
                }
            }
    return best;
}
static void full_batch(int L, const std::vector<int>& NTs, int kt, int R, int sms, int cap, int* W, int* Ct)
{
    double best = 1e300;
    for (int ct = 1; ct <= 32; ++ct)
        for (int w : WS) {
            const int threads = 32 * w * ct;
            if (threads > LANE_THREADS || (w > units_of(L) && w > 1)) break;
            int64_t smem = 0, ctas = 0;
            bool ok = true;
            std::vector<LaneShape> s(NTs.size());
            for (size_t i = 0; ok && i < NTs.size(); ++i) {
                ok = lane_fill(L, NTs[i], kt, R, w, ct, cap, &s[i]);
                if (!ok) break;
                smem = std::max<int64_t>(smem, lane_layout(L, NTs[i], kt, s[i].gr, s[i].G, false).bytes);
                ctas += (R + s[i].gr * s[i].G - 1) / (s[i].gr * s[i].G);
            }
            if (!ok) continue;
            const int k = (int)std::min<int64_t>(lane_counted(threads, smem), (ctas + sms - 1) / sms);
            double t = 0.0, longest = 0.0;
            for (size_t i = 0; i < NTs.size(); ++i) {
                const double one = lane_clocks(L, NTs[i], s[i], k);
                t += one / k * ((R + s[i].gr * s[i].G - 1) / (s[i].gr * s[i].G));
                longest = std::max(longest, one);
            }
            t = std::max(t / sms, longest);
            t = 0.5 * (t + std::max(t, longest * (double)((ctas + (int64_t)k * sms - 1) / ((int64_t)k * sms))));
            if (t < best * 0.999) { best = t; *W = w; *Ct = ct; }
        }
}
int main()
{
    std::mt19937 g(11);
    auto U = [&](int a, int b) { return a + (int)(g() % (unsigned)(b - a + 1)); };
    int bad = 0;
    for (int i = 0; i < 3000; ++i) {
        const int L = U(1, 16), NT = U(1, 64), R = 1 + (int)std::exp(std::log(1000.0) * (g() % 1000) / 1000.0), n = U(1, 16);
        const int kt = U(0, 3) ? 19 : 4 * U(5, 32);
        const bool walk = n == 1 && U(0, 1);
        const LaneShape a = lane_plan(L, NT, kt, R, n, walk, 152, 232432), b = full_plan(L, NT, kt, R, n, walk, 152, 232432);
        if (a.W != b.W || a.gr != b.gr || a.G != b.G || a.span != b.span) { ++bad; std::printf("plan %d %d %d %d %d\n", L, NT, kt, R, n); }
    }
    for (int i = 0; i < 300; ++i) {
        const int L = U(1, 16), n = U(1, 60), lo = U(1, 50), width = U(0, 64 - lo), R = U(1, 40), kt = U(0, 3) ? 19 : 60;
        std::vector<int> v;
        for (int j = 0; j < n; ++j) v.push_back(lo + U(0, width));
        int a = 0, b = 0, c = 0, d = 0;
        lane_plan_batch(L, v, kt, R, 152, 232432, &a, &b);
        full_batch(L, v, kt, R, 152, 232432, &c, &d);
        if (a != c || b != d) { ++bad; std::printf("batch %d %d %d %d\n", L, n, lo, R); }
    }
    std::printf("differences %d\n", bad);
}
"""


def test_plan_equals_the_full_search(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "plan.cpp", tmp_path / "plan"
    src.write_text(DRIVER)
    subprocess.run([gxx, "-std=c++17", "-O2", "-w", f"-I{CSRC}", str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout
    assert out.endswith("differences 0\n"), out[-500:]

"""The stiff integrator's shared-memory LU with a team of four warps on one matrix (csrc/stiff_lu.cuh), on the host
under ThreadSanitizer: 128 threads stand for the lanes, barriers for the warp shuffles and the team's barrier.
No two accesses of the matrix may race (a warp that still searches a column while another swaps
its rows misses the pivot, returns alone and leaves the team waiting), every thread reaches the same verdict, and
the factors are those of a lone warp, bit for bit. Rows are permuted so that every column swaps."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2312_05800_gb300", "csrc")

HARNESS = r"""
#include <pthread.h>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <thread>
#include <vector>
#define __device__
static pthread_barrier_t warp_bar[4], team_bar;
static double slots[4][32];
static thread_local int t_warp, t_lane;
template <class T> T __shfl_xor_sync(unsigned, T v, int o) {
    slots[t_warp][t_lane] = (double)v;
    pthread_barrier_wait(&warp_bar[t_warp]);
    const T r = (T)slots[t_warp][t_lane ^ o];
    pthread_barrier_wait(&warp_bar[t_warp]);
    return r;
}
#include "stiff_lu.cuh"
template <int W> struct Team {
    static constexpr int kWarps = W;
    int wt;
    void sync() const { pthread_barrier_wait(W == 1 ? &warp_bar[t_warp] : &team_bar); }
    bool lead() const { return W == 1 || wt == 0; }
};
template <int W> std::vector<double> run(std::vector<double> G, int n, int expect) {
    std::vector<double> inv(n, 0.0);
    std::vector<int> piv(n, -1);
    std::vector<int> verdict(32 * W, -1);
    std::vector<std::thread> th;
    for (int w = 0; w < W; ++w)
        for (int l = 0; l < 32; ++l)
            th.emplace_back([&, w, l] {
                t_warp = w;
                t_lane = l;
                verdict[32 * w + l] = chemgb::lu_factor<Team<W>, double>(piv.data(), G.data(), inv.data(), Team<W>{w}, l, n);
            });
    for (auto &t : th) t.join();
    for (int v : verdict)
        if (v != expect) { std::printf("verdict %d, expected %d\n", v, expect); std::exit(1); }
    G.insert(G.end(), inv.begin(), inv.end());
    for (int p : piv) G.push_back(p);
    return G;
}
int main(int argc, char **argv) {
    const int n = std::atoi(argv[1]), singular = std::atoi(argv[2]);
    for (auto &b : warp_bar) pthread_barrier_init(&b, nullptr, 32);
    pthread_barrier_init(&team_bar, nullptr, 128);
    // a diagonally dominant matrix with its rows rotated, so that each column's pivot lies further down
    std::vector<double> G((size_t)n * n);
    unsigned s = 12345;
    for (int i = 0; i < n; ++i)
        for (int j = 0; j < n; ++j) {
            s = s * 1664525u + 1013904223u;
            G[(size_t)((i + n - 7) % n) * n + j] = (s >> 8) / 16777216.0 - 0.5 + (i == j ? n : 0.0);
        }
    if (singular)
        for (int i = 0; i < n; ++i) G[(size_t)i * n + n / 2] = 0.0;
    const auto a = run<1>(G, n, !singular), b = run<4>(G, n, !singular);
    if (!singular && std::memcmp(a.data(), b.data(), a.size() * sizeof(double))) { std::printf("factors differ\n"); return 1; }
    std::printf("clean\n");
    return 0;
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    d = tmp_path_factory.mktemp("lu")
    src, exe = d / "lu.cc", d / "lu"
    src.write_text(HARNESS)
    cmd = ["g++", "-std=c++17", "-O1", "-g", "-fsanitize=thread", "-Wno-unknown-pragmas", "-I" + CSRC, str(src), "-o",
           str(exe), "-pthread"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if "tsan" in r.stderr:
        pytest.skip("no ThreadSanitizer runtime for g++ here")
    assert r.returncode == 0, r.stderr
    return str(exe)


@pytest.mark.parametrize("n,singular", [(33, 0), (54, 0), (64, 0), (54, 1)])
def test_team_lu_has_no_race(harness, n, singular):
    # a fixed address layout, which ThreadSanitizer's shadow needs on some kernels
    r = subprocess.run(["setarch", "-R", harness, str(n), str(singular)], capture_output=True, text=True, timeout=300,
                       env=dict(os.environ, TSAN_OPTIONS="halt_on_error=1"))
    if "unexpected memory mapping" in r.stderr:
        pytest.skip("ThreadSanitizer cannot map its shadow here")
    assert r.returncode == 0 and r.stdout.strip() == "clean", r.stdout + r.stderr[:4000]

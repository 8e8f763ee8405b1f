"""The register transforms of the float phases (ks_reg.cuh) on the CPU: each team's threads run as
host threads over the same exchange buffer, and every element of every length, in both directions,
has the bits that the items' transform (fft_batch) gives.  Guard values around the buffers show a
store out of range."""
import shutil
import subprocess

import pytest

from paper_2007_06427_gb300 import build as B

PROG = r"""
#include <cmath>
#include <cstdio>
#include <cstring>
#include <condition_variable>
#include <mutex>
#include <random>
#include <thread>
#include <vector>
#define KS_HOST_EMULATION 1
#include "ks_reg.cuh"
using namespace ks;
static std::mutex mu;
static std::condition_variable cv;
static int team = 1, waiting = 0, phase = 0;
namespace ks {
void rg_host_sync() {
    std::unique_lock<std::mutex> l(mu);
    const int ph = phase;
    if (++waiting == team) {
        waiting = 0;
        ++phase;
        cv.notify_all();
    } else {
        cv.wait(l, [&] { return phase != ph; });
    }
}
}
static std::vector<cpx<float>> tw(NMAX);
template <int LG, int DIR>
int check() {
    constexpr int N = 1 << LG, T = RgShape<LG>::T, ST = RgShape<LG>::STRIDE;
    std::vector<rgv> tab(rg_len(LG)), x(ST + 8, rgv{7.f, 7.f});
    for (int e = 0; e < rg_len(LG); ++e) {
        int t, m;
        rg_entry(LG, e, t, m);
        const cpx<float> w = tw[t * (NMAX / m)];
        tab[e] = rgv{w.x, w.y};
    }
    std::mt19937 g(LG);
    std::normal_distribution<float> d;
    std::vector<cpx<float>> in(N), a, b(N), out(N);
    for (auto& v : in) v = mk<float>(d(g), d(g));
    a = in;
    const cpx<float>* ref = fft_batch<float>(a.data(), b.data(), LG, 1, DIR, tw.data());
    team = T;
    std::vector<std::thread> th;
    for (int id = 0; id < T; ++id)
        th.emplace_back([&, id] {
            cpx<float> v[16];
            for (int s = 0; s < 16; ++s) v[s] = in[id + T * s];
            rg_fft<LG, DIR>(v, id, x.data() + 4, tab.data());
            for (int s = 0; s < 16; ++s) out[id + T * s] = v[s];
        });
    for (auto& t : th) t.join();
    int bad = std::memcmp(out.data(), ref, N * sizeof(cpx<float>)) != 0;
    for (int i = 0; i < 4; ++i) bad += 2 * (x[i].x != 7.f || x[ST + 4 + i].x != 7.f);
    return bad;
}
int main() {
    for (int t = 0; t < NMAX; ++t) {
        const double a = 2 * M_PI * t / NMAX;
        tw[t] = mk<float>((float)std::cos(a), (float)std::sin(a));
        if (t % 256 == 0) tw[t] = mk<float>(std::round(tw[t].x), std::round(tw[t].y));
    }
    std::printf("%d %d %d %d %d %d\n", check<5, 1>(), check<6, 1>(), check<7, 1>(), check<8, 1>(), check<9, 1>(),
                check<10, 1>());
    std::printf("%d %d %d %d %d %d\n", check<5, -1>(), check<6, -1>(), check<7, -1>(), check<8, -1>(),
                check<9, -1>(), check<10, -1>());
}
"""


def test_register_transforms_have_the_items_bits(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    (tmp_path / "reg.cpp").write_text(PROG)
    exe = tmp_path / "reg"
    # -ffp-contract=off: the fused operations are the ones the source names
    subprocess.run([cxx, "-std=c++17", "-O1", "-w", "-pthread", "-ffp-contract=off", "-I", B.CSRC,
                    str(tmp_path / "reg.cpp"), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=120).stdout
    assert out.split() == ["0"] * 12, out

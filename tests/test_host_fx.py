"""The fixed-point double transforms (ks_fx.cuh), compiled as host code, against a long double DFT.

Bound per element, with S the sum of the inputs' moduli: the scale's unit is at most
2 * 9/8 * 1.12 * 2^-63 S (the power of two, the margin, max + min/2 against the modulus).  An
input is truncated by less than one unit per component; a twiddle product is off by less than 5
(four floors of weight 2, centred, and the dropped low product), and of the inputs of a radix-4
butterfly three are multiplied.  In the worst case all of it adds up: sqrt(2) n from the input and
3/4 * 5 sqrt(2) n (1/1 + 1/4 + ...) < 7.1 n from the products of the passes, n / 4^p of which reach
an output from pass p from the end.  Then the rounding of the result, 2^-53 of it per component."""
import shutil
import subprocess

import pytest

from paper_2007_06427_gb300 import build as B

PROG = r"""
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>
#define KS_HOST_EMULATION 1
#include "ks_items.cuh"
using namespace ks;
int main(int, char** v) {
    const int lg = atoi(v[1]), mode = atoi(v[2]), n = 1 << lg;
    const double amp = atof(v[3]);
    std::vector<cpx<double>> tw(NMAX);
    for (int t = 0; t < NMAX; ++t) {
        const long double a = 2 * M_PIl * t / NMAX;
        tw[t] = {(double)cosl(a), (double)sinl(a)};
        if (t % 256 == 0) tw[t] = {std::round(tw[t].x), std::round(tw[t].y)};
    }
    std::mt19937_64 g(17);
    std::normal_distribution<double> N;
    double worst = 0, e1 = 0, e2 = 0;
    std::vector<long double> cs(n), sn(n);
    for (int t = 0; t < n; ++t) {
        cs[t] = cosl(2 * M_PIl * t / n);
        sn[t] = sinl(2 * M_PIl * t / n);
    }
    for (int rep = 0; rep < 6; ++rep)
        for (int dir = -1; dir <= 1; dir += 2) {
            const int cnt = 3;  // three transforms of different scale
            std::vector<cpx<double>> x(cnt * n), a, b(cnt * n), c, d(cnt * n);
            for (int i = 0; i < cnt * n; ++i) {
                const int m = i % n, k = std::min(m, n - m);
                double w = amp * std::pow(1e3, i / n);
                if (mode == 1) w *= k <= n / 3 ? std::exp(-k / 2.0) : 0;   // a band, decaying
                if (mode == 2) w *= k <= n / 3 ? std::exp(-k / 8.0) : 0;
                if (mode == 3) w *= m == (7 * rep + 1) % n;                // one mode
                x[i] = {N(g) * w, N(g) * w};
            }
            a = x;
            c = x;
            int sc[cnt];
            const cpx<double>* r = fft_fx(a.data(), b.data(), lg, cnt, dir, tw.data(), sc);
            const cpx<double>* q = fft_batch<double>(c.data(), d.data(), lg, cnt, dir, tw.data());
            for (int f = 0; f < cnt; ++f) {
                long double S = 0;
                for (int m = 0; m < n; ++m) S += hypotl(x[f * n + m].x, x[f * n + m].y);
                for (int k = 0; k < n; ++k) {
                    long double sr = 0, si = 0;
                    for (int m = 0; m < n; ++m) {
                        const int t = (int)((long long)m * k % n);
                        const long double cc = cs[t], ss = dir * sn[t];
                        sr += x[f * n + m].x * cc - x[f * n + m].y * ss;
                        si += x[f * n + m].x * ss + x[f * n + m].y * cc;
                    }
                    const long double unit = ldexpl(2 * 1.125L * 1.12L * S, -63);
                    const long double tol = ldexpl(hypotl(sr, si), -53) + 8.6L * n * unit;
                    const long double e = hypotl(r[f * n + k].x - sr, r[f * n + k].y - si);
                    worst = std::max(worst, (double)(e / tol));
                    e1 += (double)(e * e / (S * S));
                    e2 += std::pow((double)(hypotl(q[f * n + k].x - sr, q[f * n + k].y - si) / S), 2);
                }
            }
        }
    std::printf("%.6g %.6g\n", worst, std::sqrt(e1 / e2));
    // zeros, infinities and NaN
    std::vector<cpx<double>> a(n, mk<double>(0, 0)), b(n);
    int sc[1];
    cpx<double>* r = fft_fx(a.data(), b.data(), lg, 1, 1, tw.data(), sc);
    int bad = 0;
    for (int k = 0; k < n; ++k) bad += !(r[k].x == 0 && r[k].y == 0);
    for (double x : {(double)INFINITY, -(double)INFINITY, (double)NAN}) {
        for (int k = 0; k < n; ++k) a[k] = mk<double>(1.0, 2.0);
        a[n - 2].y = x;
        r = fft_fx(a.data(), b.data(), lg, 1, -1, tw.data(), sc);
        for (int k = 0; k < n; ++k) bad += !(r[k].x != r[k].x && r[k].y != r[k].y);
    }
    std::printf("%d\n", bad);
    return 0;
}
"""


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("fx")
    (d / "fx.cpp").write_text(PROG)
    subprocess.run([cxx, "-std=c++17", "-O2", "-w", "-I", B.CSRC, str(d / "fx.cpp"), "-o", str(d / "fx")],
                   check=True)
    return str(d / "fx")


@pytest.mark.parametrize("mode", [0, 1, 2, 3])
@pytest.mark.parametrize("lg", range(3, 11))
def test_error_bound(exe, lg, mode):
    for amp in ("1", "0.7", "1e-200", "1e200", "1e-35", "1e33"):   # the last four leave the float range
        out = subprocess.run([exe, str(lg), str(mode), amp], check=True, capture_output=True,
                             text=True).stdout.split()
        worst, ratio, bad = float(out[0]), float(out[1]), int(out[2])
        assert worst <= 1.0, (amp, worst)
        assert bad == 0
        if mode != 3:  # random inputs: no further off than radix-4 passes in double
            assert ratio <= 1.0, (amp, ratio)

"""The twiddle products of the fixed-point transforms (fx_mul of ks_fx.cuh), compiled as host code,
against exact 128-bit products of the same integers and twiddle words, component by component.

Bounds in units of the result.  The product of the two low words, left out, is at most
|l_a l_w| + |l_b l_w'| <= 2 * 2^62 2^-63 = 1.  Rounded sums (FINE): half a unit more, and the two
bits that each of two low words loses, less than 2 * 3 * 2^-31.  By high words: four floors, each
within a unit and of weight 2, centred (or of opposite signs): 4 more.  Random operands reach every
pair of low words, those whose sum with the rounding constant leaves 32 bits among them."""
import shutil
import subprocess

import pytest

from paper_2007_06427_gb300 import build as B

PROG = r"""
#include <cstdio>
#include <random>
#define KS_HOST_EMULATION 1
#include "ks_items.cuh"
using namespace ks;
typedef __int128 I;
int main() {
    std::mt19937_64 g(5);
    double fine = 0, coarse = 0;
    for (int i = 0; i < 400000; ++i) {
        const long double a = 1.5707963267948966L * (long double)(g() >> 1) / 0x1p63L;
        const fxw w = fx_words(cosl(a), sinl(a));
        const fxc v{(long long)g() / 2, (long long)g() / 2};  // |v| < 2^63
        const I wr = ((I)w.rh << 32) + w.rl, wi = ((I)w.ih << 32) + w.il;  // the negated twiddle, 2^-63
        const I x = (I)v.y * wi - (I)v.x * wr, y = -(I)v.x * wi - (I)v.y * wr;
        auto off = [&](fxc p) {
            const double e = (double)(x - ((I)p.x << 63)) * 0x1p-63, f = (double)(y - ((I)p.y << 63)) * 0x1p-63;
            return std::max(std::fabs(e), std::fabs(f));
        };
        fine = std::max(fine, off(fx_mul<true>(v, w)));
        coarse = std::max(coarse, off(fx_mul<false>(v, w)));
    }
    std::printf("%.9g %.9g\n", fine, coarse);
}
"""


def test_products_within_their_bounds(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    (tmp_path / "mul.cpp").write_text(PROG)
    subprocess.run([cxx, "-std=c++17", "-O2", "-w", "-I", B.CSRC, str(tmp_path / "mul.cpp"), "-o",
                    str(tmp_path / "mul")], check=True)
    out = subprocess.run([str(tmp_path / "mul")], check=True, capture_output=True, text=True).stdout
    fine, coarse = map(float, out.split())
    assert fine <= 1.5 + 3 * 2.0**-30
    assert coarse <= 5.0

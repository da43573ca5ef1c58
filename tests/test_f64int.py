"""The integer forms of float64 subtraction and multiplication (f64int.cuh) give
the hardware's bits over the ranges they state: random operands, neighbours,
exact ties of the rounding, equal operands and zeros (compiled for the host)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
HEADER = os.path.join(os.path.dirname(HERE), "paper_2404_07183_gb300", "csrc", "f64int.cuh")

SOURCE = r'''
#include "%s"
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
using namespace pcfgb;
static uint64_t bits(double x) { uint64_t u; memcpy(&u, &x, 8); return u; }
static double value(uint64_t u) { double x; memcpy(&x, &u, 8); return x; }
int main()
{
    std::mt19937_64 r(%d);
    long widths = 0, products = 0, bad = 0;
    for (long i = 0; i < 3000000; ++i) {
        double t = ldexp(1.0 + (r() >> 12) * 0x1p-52, (int)(r() %% 40) - 20), c = t;
        switch (i %% 6) {
        case 0: c = t * ((r() >> 11) * 0x1p-53); break;
        case 1: c = value(bits(t) - r() %% (1ull << (r() %% 53))); break;
        case 2: break;                                               // equal
        case 3: t = ldexp((double)(r() %% 1000000), -(int)(r() %% 10));
                c = ldexp((double)(r() %% 1000000), -(int)(r() %% 10)); break;
        case 4: t = ldexp((double)((1ull << 52) | (r() & kMant)), 1 + r() %% 10);   // ties
                c = (double)((1ull << 52) | (r() & kMant)); break;
        default: t = value(r() & 0x7fffffffffffffffull); c = value(r() & 0x7fffffffffffffffull);
                 if (!(t < 1e308) || !(c < 1e308)) continue;
        }
        if (c > t) std::swap(t, c);
        const uint64_t n = bits(t), k = bits(c);
        const uint32_t e = (uint32_t)(n >> 52);
        if (c > 0 && e >= kWidthExpLo && e <= kWidthExpHi && k >= n - ((uint64_t)kWidthOctaves << 52)) {
            ++widths;
            bad += f64i_width(n, k) != bits(t - c);
        }
        double a = (r() & 1) ? t : -t, b = (r() & 1) ? c : -c;
        if ((i & 63) == 7) b = (r() & 1) ? 0.0 : -0.0;
        if ((i & 127) == 9) b = a;
        if (f64i_value_suits(bits(a)) && f64i_value_suits(bits(b))) {
            volatile double p = a * b, d = a - b;
            volatile double q = d * d;
            products += 2;
            bad += f64i_mul(bits(a), bits(b)) != bits(p);
            bad += f64i_mul(bits(d), bits(d)) != bits(q);
        }
    }
    printf("%%ld %%ld %%ld\n", widths, products, bad);
    return 0;
}
'''


@pytest.mark.parametrize("seed", [1, 2])
def test_bits_equal_the_hardware(tmp_path, seed):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SOURCE % (HEADER, seed))
    subprocess.run([gxx, "-O1", "-ffp-contract=off", "-o", str(exe), str(src)], check=True)
    widths, products, bad = map(int, subprocess.run([str(exe)], capture_output=True, text=True,
                                                    check=True).stdout.split())
    assert widths > 1000000 and products > 2000000 and bad == 0

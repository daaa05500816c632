"""FP32 <-> FP64 by integer operations (csrc/fp_convert.h) against the conversions of the language, on the CPU:
every exponent, both signs, mantissas at the rounding points, zeros, denormals, infinities and NaN."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_21869_gb300", "csrc")

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include "fp_convert.h"
static uint64_t seed = 88172645463325252ull;
static uint64_t next() { seed ^= seed << 13; seed ^= seed >> 7; seed ^= seed << 17; return seed; }
template <class B, class T> bool same(T a, T b) { return (std::isnan(a) && std::isnan(b)) || same_bits<B>(a) == same_bits<B>(b); }
int main() {
    long n = 0, bad = 0;
    auto wide = [&](uint32_t u) {
        const float x[2] = {1.0f, same_bits<float>(u)};
        double y[2];
        widened(x, y);
        ++n;
        bad += !same<uint64_t>(y[1], (double)x[1]) || y[0] != 1.0;
    };
    auto narrow = [&](uint64_t u) {
        const double x[2] = {same_bits<double>(u), -1.0};
        float y[2];
        narrowed(x, y);
        ++n;
        bad += !same<uint32_t>(y[0], (float)x[0]) || y[1] != -1.0f;
    };
    for (uint32_t s = 0; s < 2; ++s) {
        for (uint32_t e = 0; e < 256; ++e)
            for (int m = 0; m < 300; ++m) {
                const uint32_t k = m < 4 ? m : (m < 8 ? 0x7fffffu - (m - 4) : (uint32_t)next() & 0x7fffffu);
                wide((s << 31) | (e << 23) | k);
            }
        for (uint64_t e = 0; e < 2048; ++e)
            for (int m = 0; m < 300; ++m) {
                uint64_t k = next() & 0xfffffffffffffull;
                if (m < 60) k = (k & ~0x1fffffffull) | (0x10000000ull + (m % 5) - 2);   // about half a unit
                else if (m < 80) k = (k & ~0x1fffffffull) | ((m % 3) ? m % 3 - 1 : 0x1fffffffull);
                else if (m < 90) k = 0xfffffffffffffull - (next() & 0x1fffffffull);     // rounds into the next exponent
                narrow((s << 63) | (e << 52) | k);
            }
    }
    printf("%ld cases, %ld wrong\n", n, bad);
    return bad != 0;
}
"""


def test_conversions_equal_the_languages(tmp_path):
    src, exe = tmp_path / "convert.cpp", tmp_path / "convert"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout

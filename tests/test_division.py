"""The division by a repeated divisor (csrc/esp_div.h, Markstein's two correction steps) gives the hardware's
correctly rounded quotient for every operand the price update feeds it: excess demands (whole numbers below
2^63 in magnitude) and prices (zero, or 2^-900 to 2^1000) over capacities (whole numbers in [1, 2^63)).
"""

import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

DRIVER = r"""
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <initializer_list>
#include "esp_div.h"
static uint64_t s = 88172645463325252ull;
static uint64_t rnd() { s ^= s << 13; s ^= s >> 7; s ^= s << 17; return s; }
static double bits(uint64_t b) { double d; std::memcpy(&d, &b, 8); return d; }
static uint64_t word(double d) { uint64_t b; std::memcpy(&b, &d, 8); return b; }
int main()
{
    long bad = 0;
    for (long i = 0; i < 6000000; ++i) {
        // capacities: any number of bits, and neighbours of powers of two
        uint64_t c = (rnd() >> 1) >> (rnd() % 62);
        if (i % 5 == 0)
            c = (1ull << (rnd() % 63)) + (rnd() % 5) - 2;
        c = c < 1 || c >> 63 ? 1 : c;
        const double b = (double)(int64_t)c, y = 1.0 / b;
        int64_t e = (int64_t)(rnd() >> (1 + rnd() % 62)) * (rnd() & 1 ? 1 : -1);
        if (i % 7 == 0)
            e = (int64_t)c * (int64_t)(rnd() % 3) + (int64_t)(rnd() % 3) - 1;   // quotients at and next to whole numbers
        const double a = (double)e;
        bad += word(esp::div_by(a, b, y)) != word(a / b);
        // prices: random significands and exponents inside div_safe's range, and values next to multiples of b
        double p = bits((rnd() >> 12) | ((123 + rnd() % 1900) << 52));
        if (i % 3 == 0) {
            p = b * (1.0 + (double)(rnd() % 64) / 64.0);
            p = bits(word(p) + rnd() % 5 - 2);
        }
        if (i % 1000 == 0)
            p = 0.0;
        if (esp::div_safe((long long)word(p)))
            bad += word(esp::div_by(p, b, y)) != word(p / b);
        else
            ++bad;
    }
    for (double p : {5e-324, 1e-300, bits(123ull << 52) * 0.99, bits(2023ull << 52), 1.7976931348623157e308})
        bad += esp::div_safe((long long)word(p));
    std::printf("%ld\n", bad);
    return 0;
}
"""


def test_division_by_a_repeated_divisor_is_correctly_rounded(tmp_path):
    src, exe = tmp_path / "d.cpp", tmp_path / "d"
    src.write_text(DRIVER)
    csrc = os.path.join(ROOT, "paper_2608_07971_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-I", csrc, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.strip() == "0"

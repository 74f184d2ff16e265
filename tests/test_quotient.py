"""quot.cuh's division by a known reciprocal against the division, bit for bit, on
the host: random quotients, quotients as close to a rounding boundary as 53 bits
allow (a 2^54 = b (2Q + 1) + s with |s| <= 3), and the dividends that need care;
quotients below 2^-900 within two ulp."""
import subprocess

from paper_2608_24348_gb300 import build

SRC = r"""
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <limits>
#include <random>
#include "quot.cuh"
static long bad[3], seen[3];
static void check(int kind, double a, double b)
{
    const double x = div_r(a, b, 1.0 / b), y = a / b;
    ++seen[kind];
    if (std::isnan(x) && std::isnan(y)) return;
    if (std::fabs(y) > 0 && std::fabs(y) < 0x1p-900)
        bad[kind] += !(std::fabs(x - y) <= std::fmax(2 * 0x1p-52 * std::fabs(y), 1e-323));
    else if (memcmp(&x, &y, sizeof x))
        ++bad[kind];
}
int main()
{
    std::mt19937_64 g(1);
    for (int i = 0; i < 400000; ++i) {
        const double b = ldexp(1 + (g() >> 12) * 0x1p-52, (int)(g() % 40) - 20);
        check(0, ldexp(1 + (g() >> 12) * 0x1p-52, (int)(g() % 80) - 40) * (g() & 1 ? 1 : -1), b);
    }
    for (int i = 0; i < 100000; ++i) {
        const uint64_t B = (g() >> 11) | (1ull << 52) | 1, M = (1ull << 54) - 1;
        uint64_t inv = B;  // of B modulo 2^64
        for (int k = 0; k < 6; ++k) inv *= 2 - B * inv;
        for (int s = -3; s <= 3; s += 2) {
            const uint64_t o = ((uint64_t)(-(int64_t)s) * inv) & M;  // 2Q + 1
            const unsigned __int128 p = (unsigned __int128)B * o + (__int128)s;
            const uint64_t A = (uint64_t)(p >> 54);
            if (!(o >> 53) || ((uint64_t)p & M) || (A >> 52) != 1) continue;
            check(1, (double)A, (double)B);
        }
    }
    const double inf = std::numeric_limits<double>::infinity();
    const double as[] = {0.0, -0.0, inf, -inf, std::nan(""), 5e-324, -1e-310, 2.3e-308, 1e-250, 1e250, 1.7e308, -1.7e308, 1.0};
    const double bs[] = {1e-3, 0.3, 1.0, 3.0, 7e5};
    for (double a : as)
        for (double b : bs) check(2, a, b);
    for (int k = 0; k < 3; ++k) printf("%ld %ld\n", seen[k], bad[k]);
}
"""


def test_quotients_are_those_of_the_division(tmp_path):
    src, exe = tmp_path / "q.cpp", tmp_path / "q"
    src.write_text(SRC.replace('#include "quot.cuh"', '#include <string.h>\nusing std::fma;\n#include "quot.cuh"'))
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I", build.CSRC, str(src), "-o", str(exe)],
                   check=True, capture_output=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    seen, bad = [int(v) for v in out[0::2]], [int(v) for v in out[1::2]]
    assert seen[0] == 400000 and seen[1] > 50000 and seen[2] == 65
    assert bad == [0, 0, 0]

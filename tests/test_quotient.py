"""csrc/quotient.h against the division it stands for, on the host: fused
multiply-adds round alike on both machines."""
import subprocess

from tests.test_host_logic import CSRC

SOURCE = r"""
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <random>
#include "quotient.h"
using namespace nnqp;
typedef unsigned __int128 u128;
static long bad, tested;
static double bits(uint64_t m, int e, bool neg) { return (neg ? -1.0 : 1.0) * ldexp((double)m, e - 52); }
static void check(double a, double b) {
    if (a != 0.0 && !(fabs(a) >= ldexp(1.0, -400) && fabs(a) < ldexp(1.0, 400))) return;
    if (!(fabs(b) > 1e-180 && fabs(b) < 1e180)) return;
    ++tested;
    const double x = quotient(a, b, 1.0 / b), t = a / b;
    if (!(x == t)) {
        if (++bad <= 5) printf("%a / %a: %a, not %a\n", a, b, x, t);
    }
}
static uint64_t half_power(uint64_t b, int k) {   // 2^-k mod b, b odd
    const uint64_t h = (b + 1) / 2;
    u128 r = 1;
    for (int i = 0; i < k; ++i) r = r * h % b;
    return (uint64_t)r;
}
int main() {
    std::mt19937_64 g(7);
    const uint64_t one = 1ull << 52;
    auto some = [&](int kind) {   // significands: any, near 2, near 1
        const uint64_t w = g() % (1ull << (1 + g() % 51));
        return kind == 0 ? one | (g() & (one - 1)) : kind == 1 ? 2 * one - 1 - w : one + w;
    };
    for (long i = 0; i < 4000000; ++i) {
        const int ea = (int)(g() % 799) - 399, eb = (int)(g() % 1195) - 597;
        check(bits(some(i % 3), ea, g() & 1), bits(some(i / 3 % 3), eb, g() & 1));
    }
    // quotients next to the middle of two numbers: a 2^k = s (mod b), s small
    for (long i = 0; i < 60000; ++i) {
        const uint64_t b = some(i % 3) | 1;
        if (b >> 53) continue;
        for (int k = 53; k <= 54; ++k) {
            const uint64_t iv = half_power(b, k);
            for (int s = -4; s <= 4; ++s) {
                const uint64_t r = (uint64_t)((u128)(s < 0 ? b + s : (uint64_t)s) * iv % b);
                for (int c = 0; c < 2; ++c) {
                    const uint64_t a = r + (c ? b : 0);
                    if (a > 0 && a < 2 * one) check((double)a, (double)b);
                }
            }
        }
    }
    const double special[] = {0.0, -0.0, 1.0, -1.0, 3.0, 1e120, -1e-120, 3e-121, 2.5e120, 1e-180, 1e180};
    for (double a : special)
        for (double b : special) check(a, b);
    printf("%ld of %ld differ\n", bad, tested);
    return bad != 0;
}
"""


def test_quotients_are_the_rounded_ones(tmp_path):
    src, exe = tmp_path / "q.cpp", tmp_path / "q"
    src.write_text(SOURCE)
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC, str(src), "-o", str(exe)])
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout

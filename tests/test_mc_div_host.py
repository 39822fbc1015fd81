"""The tree search's division (mc_div in csrc/trigram.cu), compiled for the host, where fused multiply-add and the operator round as on the
device: for every divisor that a search can have, the operator's quotient, bit for bit."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
SOURCE = os.path.join(os.path.dirname(HERE), "paper_2407_12021_b200", "csrc", "trigram.cu")

PROGRAM = r"""
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <initializer_list>
#include <limits>
static bool by_operator;
static int __double2hiint(double v) { uint64_t b; memcpy(&b, &v, 8); return (int)(b >> 32); }
static double __ddiv_rn(double a, double b) { by_operator = true; return a / b; }
static double __dmul_rn(double a, double b) { return a * b; }
static double __fma_rn(double a, double b, double c) { return std::fma(a, b, c); }
%s
static uint64_t state = 1;
static uint64_t random64() {                                    // SplitMix64
    uint64_t z = (state += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
static double from_bits(uint64_t b) { double v; memcpy(&v, &b, 8); return v; }
static uint64_t bits(double v) { uint64_t b; memcpy(&b, &v, 8); return b; }
int main() {
    const double inf = std::numeric_limits<double>::infinity(), edges[] = {0.0, std::ldexp(1.0, -1074), std::ldexp(1.0, -1022), std::ldexp(1.0, -927),
        std::ldexp(1.0, 992), std::ldexp(1.0, 993), std::numeric_limits<double>::max(), inf, std::nan("")};
    long long differ = 0, fast = 0, all = 0;
    for (int n = 1; n <= %d; ++n) {
        const double rcp = 1.0 / n;
        auto check = [&](double a) {
            for (double s : {a, -a}) {
                by_operator = false;
                const double got = mc_div(s, n, rcp), want = s / n;
                ++all;
                fast += !by_operator;
                if (bits(got) != bits(want) && !(std::isnan(got) && std::isnan(want))) ++differ;
            }
        };
        for (double e : edges)
            for (double a : {std::nextafter(e, -inf), e, std::nextafter(e, inf)}) check(a);
        for (int i = 0; i < 20000; ++i) {
            check(from_bits(random64() & ~(1ull << 63)));                                                        // any exponent
            check(1.0 + (double)(random64() >> 11) * 0x1p-53 * 400.0);                                           // sums of scores
            // quotients next to a double and to the middle between two: the products of n with them, and their neighbours
            const double q = from_bits((random64() >> 12) | 0x3FF0000000000000ull);
            const double half = std::fma(q, (double)n, std::ldexp((double)n, -53));
            for (double a : {q * n, half}) { check(std::nextafter(a, 0.0)); check(a); check(std::nextafter(a, inf)); }
        }
    }
    printf("%%lld %%lld %%lld\n", differ, fast, all);
    return 0;
}
"""


def test_quotient_is_the_operators(tmp_path):
    text = open(SOURCE).read()
    start = text.index("__device__ __forceinline__ double mc_div(")
    code = text[start:text.index("\n}\n", start) + 3].replace("__device__ __forceinline__", "static")
    most = int(text.split("constexpr int MC_MAX_ITER = ")[1].split(",")[0]) + 1
    assert most == 161
    (tmp_path / "mc_div.cpp").write_text(PROGRAM % (code, most))
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", str(tmp_path / "mc_div.cpp"), "-o", str(tmp_path / "mc_div")], check=True)
    differ, fast, count = map(int, subprocess.run([str(tmp_path / "mc_div")], capture_output=True, text=True, check=True, timeout=600).stdout.split())
    assert differ == 0
    assert fast > count // 2                # the path without the operator is the one that is compared

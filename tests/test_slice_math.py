"""The Gibbs/measure kernel's exact rewritings (csrc/slice_math.h), on the host: the division by N
bit for bit against the plain one for every lattice size, and the integer threshold against u < p
at the words next to it."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2510_13866_gb300", "csrc")
MAIN = """
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <initializer_list>
using std::ceil;
using std::fma;
#include "slice_math.h"
static uint64_t state = 88172645463325252ull;
static uint64_t next() {
    state ^= state << 13;
    state ^= state >> 7;
    return state ^= state << 17;
}
int main() {
    long bad = 0, n = 0;
    for (int L : {2, 3, 4, 6, 8, 12, 16, 24, 32, 48, 64, 128}) {
        const int N = L * L;
        const double dn = N, inv = 1.0 / dn;
        const bool pow2 = (N & (N - 1)) == 0;
        for (long k = -4; k < 400000; ++k) {
            // floats of every magnitude, zero, the least and the largest one
            float x = k == -4 ? 0.f : k == -3 ? 0x1.0p-149f : k == -2 ? 0x1.fffffep+127f : k == -1 ? 1.f : 0.f;
            if (k >= 0) {
                uint32_t bits = uint32_t(next() >> 33);
                if (k % 2) bits = (bits & 0x7fffffu) | (uint32_t(100 + k % 60) << 23);  // those that occur
                if ((bits >> 23) == 255) continue;
                std::memcpy(&x, &bits, 4);
            }
            const double got = hqmc::div_n(double(x), dn, inv, pow2), want = double(x) / dn;
            bad += std::memcmp(&got, &want, 8) != 0;
            ++n;
        }
    }
    std::printf("%ld %ld\\n", n, bad);
    n = bad = 0;
    for (long k = 0; k < 400000; ++k) {
        double p = k == 0 ? 0.0 : k == 1 ? 1.0 : k == 2 ? 0x1.0p-1074 : k == 3 ? 0x1.0p-53 : k == 4 ? 0x1.8p-53 : k == 5 ? 0x1.fffffffffffffp-1 : 0.0;
        if (k > 5 && k % 2) p = 1.0 / (1.0 + std::exp(-2.0 * 0.37 * double(k % 129 - 64) * (1 + double(k) / 4e5)));
        else if (k > 5) p = std::ldexp(double(next() >> 11) * 0x1.0p-53, -int(next() % 70));
        const uint64_t thr = hqmc::gibbs_threshold(p);
        for (int d = -2; d <= 2; ++d) {
            const int64_t w = int64_t(thr) + d;
            if (w < 0 || w >= (int64_t(1) << 53)) continue;
            bad += (uint64_t(w) < thr) != (double(w) * 0x1.0p-53 < p);
            ++n;
        }
    }
    std::printf("%ld %ld\\n", n, bad);
}
"""


def test_division_and_threshold_are_exact(tmp_path):
    (tmp_path / "main.cpp").write_text(MAIN)
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-I", CSRC, "-o", str(tmp_path / "main"),
                           str(tmp_path / "main.cpp")])
    out = subprocess.run([str(tmp_path / "main")], capture_output=True, text=True, check=True).stdout.split()
    assert int(out[0]) > 4_000_000 and int(out[1]) == 0
    assert int(out[2]) > 1_000_000 and int(out[3]) == 0

"""The rule that gives a chain its window (csrc/window_rule.h), on the host: R and the least total that
a window answers for, from their definitions, at hops on both sides of each line."""
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2510_13866_gb300", "csrc")
MAIN = """
#include <cstdio>
#include <vector>
#include "window_rule.h"
int main() {
    int L;
    double wmax;
    while (std::scanf("%d %la", &L, &wmax) == 2) {
        std::vector<double> g(L);
        for (double &v : g) std::scanf("%la", &v);
        const hqmc::WinRule w = hqmc::window_rule(g.data(), L, wmax);
        std::printf("%d %a\\n", w.R, double(w.least));
    }
}
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    d = tmp_path_factory.mktemp("rule")
    (d / "main.cpp").write_text(MAIN)
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-I", CSRC, "-o", str(d / "main"), str(d / "main.cpp")])

    def call(g, wmax):
        text = f"{len(g)} {float(wmax).hex()} " + " ".join(float(v).hex() for v in g)
        R, least = subprocess.run([str(d / "main")], input=text, capture_output=True, text=True, check=True).stdout.split()
        return int(R), float.fromhex(least)

    return call


def ring(L, z):
    term = np.zeros(L)
    term[0] = 1.0
    g = term.copy()
    for n in range(1, 4 * L):
        term = (np.roll(term, 1) + np.roll(term, -1)) * (z / n)
        g += term
    return g


@pytest.mark.parametrize("L", [48, 64, 128])
@pytest.mark.parametrize("z,R", [(1 / 32, 8), (0.05, 9), (0.1, 10), (0.125, 11), (0.15, 11), (0.165, 11), (0.168, 0), (0.2, 0), (1.0, 0)])
@pytest.mark.parametrize("wmax", [1.0, 3.0])
def test_window_of_a_chain(rule, L, z, R, wmax):
    g = ring(L, z)
    got, least = rule(g, wmax)
    assert got == R
    if R == 0:
        assert least == 0.0
        return
    assert g[R + 1] <= 2.0**-60 * g[0] < g[R]
    assert abs(least - 2.0**36 * 4 * g[R + 1] * g[0] * wmax) <= 1e-6 * least
    # a site beyond R steps has at most this weight times f, and f sums to less than 2 max W
    outside = g[:, None] * g[None, :]
    d = np.minimum(np.arange(L), L - np.arange(L))
    outside[(d[:, None] <= R) & (d[None, :] <= R)] = 0.0
    assert 2.0 * wmax * outside.max() <= 2.0**-36 * least


def test_small_lattices_and_no_hopping(rule):
    assert rule(ring(24, 0.05), 1.0) == (0, 0.0)
    R, least = rule(ring(64, 0.0), 1.0)
    assert R == 1 and abs(least - 1e-30) < 1e-36

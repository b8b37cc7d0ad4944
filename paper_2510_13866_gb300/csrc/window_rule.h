// window_rule.h -- which chains draw their worldlines from windows of f (ffbs_window.cuh), and how
// wide.  Host code, without CUDA.
#pragma once

#include <algorithm>

namespace hqmc {

constexpr int kWinHalf = 12;  // half width of the window that is loaded

struct WinRule {
    int R = 0;         // steps beyond which G is negligible (0: no window)
    float least = 0.f; // the least conditional total S that the window answers for
};

// R is the least one with g(R + 1) <= 2^-60 g(0): the sites beyond it then hold less than 2^-36 of
// any total S >= least = 2^36 4 g(R + 1) g(0) max W, and `least` stays below 2^-22 of the largest
// weight, so that almost every draw is answered (t dtau = 1/32, 0.05, 0.1: R = 8, 9, 10).  Hops that
// need R > kWinHalf - 1 (t dtau above 0.165) leave no margin for the moves between load and draw: no
// window.  g: the ring's propagator, wmax: the largest W.
inline WinRule window_rule(const double *g, int L, double wmax) {
    WinRule w;
    if (L <= 2 * kWinHalf + 1) return w;
    double far = 0.0;  // the largest g beyond R
    for (int R = L / 2 - 1; R >= 1; --R) {
        far = std::max(far, g[R + 1]);
        if (far > 0x1.0p-60 * g[0]) return w;
        if (R > kWinHalf - 1) continue;
        const double m = 0x1.0p+36 * 4.0 * far * g[0] * wmax;
        if (!(m < 1e30)) return w;
        w.R = R;
        w.least = float(std::max(m, 1e-30));
    }
    return w;
}

}  // namespace hqmc

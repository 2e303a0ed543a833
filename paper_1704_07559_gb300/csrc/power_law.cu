// power_law.cu -- host side of power_law.h.
#include "power_law.h"

#include <cmath>

namespace lbm {

PowerLawGuess power_law_guess(double n, double K, double tau_min, double tau_max, double tol, int max_iter) {
    PowerLawGuess g = {};
    const double m = n - 1.0;
    if (m == 0.0 || std::fabs(m) > 0.5 || !(K > 0.0) || max_iter < 48 || !(tol <= 1e-5)) return g;
    // log2 C = v + m log2(1/2 + 2^v) rises with v = log2(tau - 1/2)
    auto lgc = [&](double v) { return v + m * std::log2(0.5 + std::exp2(v)); };
    const double v0 = std::log2(tau_min - 0.5), v1 = std::log2(tau_max - 0.5);
    const double lo = lgc(v0), hi = lgc(v1);
    if (!(hi - lo > 1e-3)) return g;
    // interpolation at the Chebyshev points of degree D, as divided differences, then as powers of x
    constexpr int D = POWER_LAW_DEGREE;
    double x[D + 1], d[D + 1], p[D + 1] = {};
    for (int i = 0; i <= D; ++i) {
        x[i] = std::cos(3.14159265358979323846 * (i + 0.5) / (D + 1));
        const double c = lo + 0.5 * (x[i] + 1.0) * (hi - lo);
        double a = v0, b = v1;
        for (int it = 0; it < 60; ++it) {
            const double mid = 0.5 * (a + b);
            (lgc(mid) < c ? a : b) = mid;
        }
        d[i] = 0.5 * (a + b);
    }
    for (int k = 1; k <= D; ++k)
        for (int i = D; i >= k; --i) d[i] = (d[i] - d[i - 1]) / (x[i] - x[i - k]);
    for (int k = D; k >= 0; --k) {
        for (int i = D; i >= 1; --i) p[i] = p[i - 1] - x[k] * p[i];
        p[0] = d[k] - x[k] * p[0];
    }
    g.on = 1;
    g.ax = float(m / (hi - lo));  // log2 C = log2 3K + (m/2) log2(2 B:B)
    g.x0 = float(2.0 * (std::log2(3.0 * K) - lo) / (hi - lo) - 1.0);
    for (int i = 0; i <= D; ++i) g.p[i] = float(p[i]);
    if (!std::isfinite(g.ax) || !std::isfinite(g.x0)) g.on = 0;
    return g;
}

}  // namespace lbm

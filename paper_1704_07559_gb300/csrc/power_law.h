// power_law.h -- first guesses of the power-law closure's tau.
//
// The closure solves tau = F(tau), F(tau) = 1/2 + 3K |S|^(n-1) clamped to [tau_min, tau_max], with
// S = A + B/tau.  On these bases the rate-free part A holds the flow's dilatation only, which is small at
// low Mach number.  Without it |S| = b/tau, b = sqrt(2 B:B), and tau is the root of
//   (tau - 1/2) tau^(n-1) = C,  C = 3K b^(n-1),
// a function of C alone for a context's n.  log2(tau - 1/2) bends only slowly over log2 C (its slope runs
// from 1 to 1/n), so between the clamps a polynomial of degree 6 gives tau to about 1e-3: the start of
// the iteration in tau_fixed_point.  (A table of 257 points is nearer, but its look-ups miss L1 among the
// streaming populations: a cavity at rest, where one sweep suffices, fell from 83.6 to 76.4 GLUPS.)
//
// F is a contraction in log tau with factor at most |n - 1|, so it has one fixed point for |n - 1| < 1.  The
// guess is used for |n - 1| <= 1/2, where plain sweeps reach any tolerance within 48 sweeps and the
// two iterations therefore end at the same root; other n, a lower sweep limit, a coarse tolerance, K = 0
// and n = 1 (F does not depend on tau) keep the plain sweeps from tau0.
#pragma once

namespace lbm {

constexpr int POWER_LAW_DEGREE = 6;

struct PowerLawGuess {
    int on;        // 0: plain sweeps from tau0 (see above)
    float ax, x0;  // x = ax log2(2 B:B) + x0: -1 at tau_min, 1 at tau_max
    float p[POWER_LAW_DEGREE + 1];  // log2(tau - 1/2) = p[0] + x (p[1] + x (p[2] + ...))
};

PowerLawGuess power_law_guess(double n, double K, double tau_min, double tau_max, double tol, int max_iter);

}  // namespace lbm

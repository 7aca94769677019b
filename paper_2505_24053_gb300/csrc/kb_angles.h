// kb_angles.h -- the Kannala-Brandt distortion's angles on the host: the vertical
// field of view and the largest invertible angle (App. E).
//
// Both are the first step of a fine grid (8192 steps to half the field of view, 4096
// to pi) that a condition holds at. Whole runs of steps where bounds of the polynomial
// rule the condition out are skipped, so that a camera takes some dozen evaluations
// where walking the grid took thousands: ~50 us a call that is given a camera, more
// than the kernels of a small render or of a resampling. The steps that remain are
// evaluated as on the full walk, so the results are the same doubles.
#pragma once

#include <algorithm>
#include <cmath>

namespace geer {

// Distorted angle phi (1 + k1 phi^2 + k2 phi^4 + k3 phi^6 + k4 phi^8).
inline double kb_theta_d(const float k[4], double phi) {
    const double p2 = phi * phi;
    return phi * (1.0 + p2 * (k[0] + p2 * (k[1] + p2 * (k[2] + p2 * k[3]))));
}

// Bounds over phi in [a, b], 0 <= a <= b: the distorted angle from above, its slope
// from below; slack: a bound on the rounding errors of either.
struct KbBounds {
    double theta_max, slope_min, slack;
};
inline KbBounds kb_bounds(const float k[4], double a, double b) {
    double pa = 1.0, pb = 1.0, up = 1.0, slope = 1.0, mag = 1.0;
    for (int j = 0; j < 4; ++j) {
        pa *= a * a;
        pb *= b * b;
        up += std::max(k[j] * pa, k[j] * pb);
        slope += (2 * j + 3) * std::min(k[j] * pa, k[j] * pb);
        mag += (2 * j + 3) * std::fabs(k[j]) * pb;
    }
    return {up > 0.0 ? b * up : a * up, slope, 1e-12 * (1.0 + b) * mag};
}

// The first step s in (s0, s1] with hit(s), else 0; none(s0, s1): no step of (s0, s1]
// can be a hit.
template <typename Hit, typename None>
int first_step(int s0, int s1, Hit hit, None none) {
    if (s1 - s0 == 1) return hit(s1) ? s1 : 0;
    if (none(s0, s1)) return 0;
    const int mid = s0 + (s1 - s0) / 2, s = first_step(s0, mid, hit, none);
    return s ? s : first_step(mid, s1, hit, none);
}

// The vertical field of view whose half maps to h / w times what fov_x / 2 maps to:
// twice the smallest root, bracketed on the grid, then bisected.
inline double kb_fov_y(const float k[4], double fov_x, double w, double h) {
    const double edge = kb_theta_d(k, 0.5 * fov_x);
    if (!(edge > 0.0)) return NAN;
    const double target = edge * h / w;
    double lo = 0.0, hi = 0.5 * fov_x;
    const int n = 8192;
    const auto at = [&](int s) { return 0.5 * fov_x * s / n; };
    const int s = first_step(0, n, [&](int i) { return kb_theta_d(k, at(i)) >= target; },
                             [&](int i, int j) {
                                 const KbBounds b = kb_bounds(k, at(i), at(j));
                                 return b.theta_max + b.slack < target;
                             });
    if (s) {
        hi = at(s);
        lo = at(s - 1);
    }
    for (int it = 0; it < 200; ++it) {
        const double mid = 0.5 * (lo + hi);
        const bool done = mid == lo || mid == hi;  // neighbours: further halving changes nothing
        if (kb_theta_d(k, mid) >= target) hi = mid; else lo = mid;
        if (done) break;
    }
    return 2.0 * hi;
}

// The first turning point of the distorted angle below pi (as far as it is increasing,
// it can be inverted), or pi.
inline double kb_phi_max(const float k[4]) {
    const int n = 4096;
    const auto at = [&](int s) { return M_PI * s / n; };
    const auto val = [&](int s) { return s ? kb_theta_d(k, at(s)) : 0.0; };
    const int s = first_step(0, n, [&](int i) { return !(val(i) > val(i - 1)); },
                             [&](int i, int j) {
                                 const KbBounds b = kb_bounds(k, at(i), at(j));
                                 return b.slope_min * (M_PI / n) > b.slack;
                             });
    return s ? at(s - 1) : M_PI;
}

}  // namespace geer

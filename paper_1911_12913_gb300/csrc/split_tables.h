// Difference weights of the split FP64 step (step_split.cu), with the metric, the
// time step and the sign folded in.  Host code.
#pragma once

#include <cmath>
#include <cstddef>
#include <vector>

namespace fdlbm {

// Weights of the mixed difference (Eq. 2.36) at one node of an axis, times `scale`,
// for velocity sign +1 or -1: {k + s, k, k - s, k - 2s}; `central`: next to a wall.
// Two identities of the exact weights hold for the rounded ones, because an error
// in them adds up over the steps: the sum is zero (else every step scales the
// population), and the difference of a linear function is `scale` times its slope
// (else populations travel at another speed: taps rounded one by one, 64^2 Taylor
// vortex in a mean flow after 1000 steps, momentum 1.6e-15 off 80-bit arithmetic,
// 9e-16 so).
// All weights are multiples of q = 2^(e - 52), 2^e <= |scale| < 2^(e + 1), or of 2q
// for a blend above 0.3, where they may exceed |scale|: then every sum below is at
// most 2^53 q and exact.
inline void split_taps(double beta, bool central, double scale, double out[4])
{
    if (central) {
        out[0] = 0.5 * scale;
        out[1] = out[3] = 0.0;
        out[2] = -0.5 * scale;
        return;
    }
    int e = 0;
    std::frexp(scale, &e);  // 2^(e - 1) <= |scale| < 2^e
    const double q = std::ldexp(1.0, e - (beta > 0.3 ? 52 : 53));
    auto on_grid = [&](double w) { return std::nearbyint(w / q) * q; };
    const double slope = on_grid(scale);
    const double m1 = on_grid(scale * (0.5 * (1.0 - beta))), p2 = on_grid(scale * (0.5 * beta));
    out[0] = m1;
    out[1] = (slope - m1) + (p2 - m1);
    out[2] = (m1 - slope) - (p2 + p2);
    out[3] = p2;
}

// The tables in the order bx, by (scale -h m, stage B), cx, cy (-dt m, stage C):
// [n][2][4] each, the two velocity signs of every node.
inline std::vector<double> make_split_tables(const std::vector<double> &mx, const std::vector<double> &my, bool wx,
                                             bool wy, double beta, double h, double dt)
{
    std::vector<double> out;
    out.reserve(16 * (mx.size() + my.size()));
    auto axis = [&](const std::vector<double> &m, bool wall, double s) {
        const int n = (int)m.size();
        for (int k = 0; k < n; ++k)
            for (int sign = 1; sign >= -1; sign -= 2) {
                // the second-order upwind tap k - 2 s would leave the domain
                const bool central = wall && (sign > 0 ? k < 2 : k > n - 3);
                double t[4];
                split_taps(beta, central, -s * m[k], t);
                out.insert(out.end(), t, t + 4);
            }
    };
    axis(mx, wx, h);
    axis(my, wy, h);
    axis(mx, wx, dt);
    axis(my, wy, dt);
    return out;
}

// Whether the centre weights of the two axes may be added into one for the
// diagonal populations: one value per axis in each stage, whose sum is exact.
inline bool split_centres_merge(const std::vector<double> &t, int nx, int ny)
{
    const double *p = t.data();
    for (int stage = 0; stage < 2; ++stage, p += 8 * ((size_t)nx + ny)) {
        const double a = p[1], b = p[8 * (size_t)nx + 1], s = a + b, r = s - a;
        if ((a - (s - r)) + (b - r) != 0.0) return false;  // the rounding error of s
        for (size_t k = 0; k < 2 * (size_t)nx; ++k)
            if (p[4 * k + 1] != a) return false;
        for (size_t k = 0; k < 2 * (size_t)ny; ++k)
            if (p[8 * (size_t)nx + 4 * k + 1] != b) return false;
    }
    return true;
}

}  // namespace fdlbm

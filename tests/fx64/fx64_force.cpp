// Very small forces.  A force far below a node's unit leaves the bits of the
// force-free collision.  One of a fraction of the unit acts, in the mean over
// random nodes, with its own strength: the x momentum gained against the
// force-free collision of the same node is the exact gain within 5 standard
// errors (taken from the sample) and the gain of half a unit of the coefficient
// of e_x (sum omega w e_x^2 / 2 = omega / (2 c^2)), to which theta is rounded.
#include "fx64_ref.h"

int main() {
    const int nodes = 40000;
    const int bad = every_set([&](const auto& m, auto set, const char* name) {
        using SET = decltype(set);
        constexpr int V = SET::R + 2 * SET::P, N = 3;
        Random rng(7);
        const double tau = std::sqrt(2 / M_PI) * 0.1, dt = 1 / (64 * m.c);
        int wrong = 0;
        // (1e-12: below the 64 bits after a mantissa's last, 1e-100: any number of them)
        for (double h : {1e-100, 1e-12, 1e-3, 0.03, 0.3}) {          // in units U_G
            double sum = 0, sq = 0;
            int differ = 0;
            for (int t = 0; t < nodes; ++t) {
                std::vector<double> f(V), a, b;
                const double d = 1e-3 * rng.gauss(), X = 1e-3 * rng.gauss(), Y = 1e-3 * rng.gauss();
                for (int i = 0; i < V; ++i) f[i] = m.w[i] * (d + m.ex[i] * X + m.ey[i] * Y + 1e-4 * rng.gauss());
                int E = 0;
                if (!collide_fx<SET, N, false>(m.consts(tau, dt, 0.0), tau, dt, f, b, E)) return 1;
                const Q ug = unit_g<SET>(E);
                const double g = double(2 * h * ug / (dt * m.c));
                if (!collide_fx<SET, N, true>(m.consts(tau, dt, g), tau, dt, f, a, E)) return 1;
                // the exact gain is linear in so small a force
                std::vector<Q> r1, r0;
                const double g1 = 1e-7;
                collide_ref<N, Q>(m, tau, dt, g1, f, r1);
                collide_ref<N, Q>(m, tau, dt, 0.0, f, r0);
                Q gain = 0, exact = 0;
                for (int i = 0; i < V; ++i) {
                    gain += (Q(a[i]) - Q(b[i])) * m.ex[i];
                    exact += (r1[i] - r0[i]) * m.ex[i];
                    differ += a[i] != b[i];
                }
                const double e = double((gain - exact * (Q(g) / Q(g1))) / ug);
                sum += e;
                sq += e * e;
            }
            const double mean = sum / nodes, err = std::sqrt((sq / nodes - mean * mean) / nodes);
            std::printf("%s h %.0e: mean error of the gain %.4f +- %.4f units, %d populations differ\n", name, h, mean, err, differ);
            const double omega = dt / (tau + 0.5 * dt);
            if (h < 1e-9 ? differ != 0 : std::fabs(mean) > 5 * err + 0.5 * omega / (m.c * m.c)) wrong = 1;
        }
        return wrong;
    });
    return bad ? 1 : 0;
}

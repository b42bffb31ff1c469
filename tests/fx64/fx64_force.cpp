// Very small forces.  A solve whose force is too small for the constants' shift is
// left to the FP64 form; where one is taken, it acts, in the mean over random
// nodes, with its own strength: the x momentum gained against the force-free
// collision of the same node is the exact gain within 5 standard errors (taken
// from the sample) and the gain of half a unit of the coefficient of e_x (sum omega
// w e_x^2 / 2 = omega / (2 c^2)), to which theta is rounded.
#include "fx64_ref.h"

int main() {
    const int nodes = 40000;
    const int bad = every_set([&](const auto& m, auto set, const char* name) {
        using SET = decltype(set);
        constexpr int V = SET::R + 2 * SET::P, N = 3;
        Random rng(7);
        const double tau = std::sqrt(2 / M_PI) * 0.1, dt = 1 / (64 * m.c);
        int wrong = 0;
        // h in units U_G; populations of a density near 1, whose unit is largest, and small ones
        struct { double h, amp; bool taken; } cases[] = {{1e-100, 1e-3, false}, {1e-12, 1e-3, false}, {1e-3, 1e-3, false},
                                                         {0.03, 1e-3, false}, {0.3, 1e-3, false}, {2.0, 0.3, false},
                                                         {7.0, 0.3, false}, {40.0, 0.3, true}};
        for (const auto& q : cases) {
            const double h = q.h;
            double sum = 0, sq = 0;
            int differ = 0, left = 0;
            for (int t = 0; t < nodes; ++t) {
                std::vector<double> f(V), a, b;
                const double d = q.amp * rng.uniform(-1, 1), X = 1e-3 * rng.gauss(), Y = 1e-3 * rng.gauss();
                for (int i = 0; i < V; ++i) f[i] = m.w[i] * (d + m.ex[i] * X + m.ey[i] * Y + 1e-4 * rng.gauss());
                int E = 0;
                if (!collide_fx<SET, N, false>(m.consts(tau, dt, 0.0), tau, dt, f, b, E)) return 1;
                const Q ug = unit_g<SET>(E);
                const double g = double(2 * h * ug / (dt * m.c));
                const fx::Consts k = m.consts(tau, dt, g);
                left += !k.ok;
                if (!k.ok) continue;
                if (!collide_fx<SET, N, true>(k, tau, dt, f, a, E)) return 1;
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
            const int n = nodes - left;
            std::printf("%s h %.0e: %d nodes of solves left to the FP64 form\n", name, h, left);
            if (q.taken && n < nodes / 2) wrong = 1;
            if (!n) continue;
            const double mean = sum / n, err = std::sqrt((sq / n - mean * mean) / n);
            std::printf("%s h %.0e: mean error of the gain %.4f +- %.4f units, %d populations differ\n", name, h, mean, err, differ);
            const double omega = dt / (tau + 0.5 * dt);
            if (h < 1e-9 ? differ != 0 : std::fabs(mean) > 5 * err + 0.5 * omega / (m.c * m.c)) wrong = 1;
        }
        return wrong;
    });
    return bad ? 1 : 0;
}

// Edges of the fixed-point range: forces up to the largest that the constants
// admit (theta = tau c g to 1/8, h = c g dt / 2 to 1/2), from relaxation times far
// below to far above the time step, densities and flow speeds up to where the
// checks end.  Every node that is taken is within the bound of fx64_driver.cpp:
// half an ulp of the result and of the target, and omega w B U_G.
#include "fx64_ref.h"

template <class SET, int N, bool FORCE, class MODEL>
static int run(const MODEL& m, const char* name) {
    constexpr int V = SET::R + 2 * SET::P;
    Random rng(7);
    int taken = 0, bad = 0;
    double worst = 0, se = 0;
    for (int a = 0; a < V; ++a) se += std::abs(m.ex[a]) + std::abs(m.ey[a]);
    const double mc = fx::set_emax<SET>();
    const double B = V / 2.0 + m.c * m.c * mc * se / 2 +
                     2 * (1 + 2 * mc + 3 * mc * mc + 4 * mc * mc * mc + 5 * std::pow(mc, 4));
    for (int t = 0; t < 30000; ++t) {
        const double Kn = std::pow(10.0, rng.uniform(-6, 2)), Ny = std::floor(std::exp(rng.uniform(0.7, 7.6)));
        const double tau = std::sqrt(2 / M_PI) * Kn, dt = 1 / (Ny * m.c);
        const double lim = std::fmin(0.125 / (tau * m.c), 1.0 / (dt * m.c));
        const double g = FORCE ? (t % 2 ? 1 : -1) * 0.999999 * lim * std::pow(10.0, rng.uniform(t % 3 ? -3 : -0.1, 0)) : 0.0;
        const fx::Consts k = m.consts(tau, dt, g);
        const double amp = std::pow(10.0, rng.uniform(-6, 0.7)), um = std::pow(10.0, rng.uniform(-6, 0.3)),
                     ne = std::pow(10.0, rng.uniform(-6, 1)), ang = rng.uniform(0, 2 * M_PI);
        const double d0 = amp * (t % 3 ? rng.gauss() : -rng.uniform(0, 1)), X = m.c * um * std::cos(ang),
                     Y = m.c * um * std::sin(ang);
        std::vector<double> f(V), out;
        const int mode = int(rng.r() % 3);          // noise; one half space; one half space of any size
        for (int a = 0; a < V; ++a) {
            const double s = m.ex[a] * X + m.ey[a] * Y;
            f[a] = mode == 0   ? m.w[a] * (d0 + s + ne * rng.gauss())
                   : mode == 1 ? m.w[a] * (d0 + ne * (s > 0 ? 1 : (s < 0 ? -1 : 0)))
                               : ne * 0.1 * (s > 0 ? rng.uniform(0, 1) : 0) / V;
        }
        int E = 0;
        if (!collide_fx<SET, N, FORCE>(k, tau, dt, f, out, E)) continue;
        ++taken;
        std::vector<Q> ref;
        collide_ref<N, Q>(m, tau, dt, g, f, ref);
        const double omega = dt / (tau + 0.5 * dt), omo = 1 - omega;
        double w = 0;
        for (int a = 0; a < V; ++a) {
            const Q bound = ldexpl(fabsl(ref[a]) + fabsl(ref[a] - Q(omo) * f[a]), -53) +
                            Q(omega * m.w[a]) * (B * unit_g<SET>(E)) + ldexpl(1.0L, -1070);
            const double e = double(fabsl(Q(out[a]) - ref[a]) / bound);
            if (!(e <= w)) w = e;
        }
        if (!(w <= 1.0) && bad++ < 2)
            std::printf("  %s N%d: error %.3g bounds at Kn %.3g Ny %g g %.3g (h %.3g, theta %.3g)\n", name, N, w, Kn, Ny, g,
                        0.5 * dt * m.c * std::fabs(g), tau * m.c * std::fabs(g));
        if (w > worst) worst = w;
    }
    std::printf("%s N%d force %d: taken %d, outside the bound %d, worst %.3g\n", name, N, int(FORCE), taken, bad, worst);
    return bad != 0 || taken < 1000;
}

int main() {
    const int bad = every_set([&](const auto& m, auto set, const char* name) {
        using SET = decltype(set);
        return run<SET, 2, true>(m, name) + run<SET, 3, true>(m, name) + run<SET, 4, true>(m, name) +
               run<SET, 2, false>(m, name) + run<SET, 3, false>(m, name) + run<SET, 4, false>(m, name);
    });
    return bad ? 1 : 0;
}

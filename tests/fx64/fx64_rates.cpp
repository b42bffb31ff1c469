// Tiny relaxation rates (Knudsen numbers up to 1e40) and populations down to
// 1e-268: the exponent of a target must not wrap.  Errors below 1e-12 of the
// populations' scale (rounding is 1e-15 of it; a wrapped exponent is off by
// hundreds of orders of magnitude).
#include "fx64_ref.h"

int main() {
    const int bad = every_set([&](const auto& m, auto set, const char* name) {
        using SET = decltype(set);
        constexpr int V = SET::R + 2 * SET::P, N = 3;
        Random rng(3);
        double worst = 0;
        for (int t = 0; t < 50000; ++t) {
            const double Kn = std::pow(10.0, rng.uniform(-2, 40)), amp = std::pow(10.0, rng.uniform(-268, -3));
            const double tau = std::sqrt(2 / M_PI) * Kn, dt = 1 / (64 * m.c);
            std::vector<double> f(V), out;
            std::vector<Q> ref;
            for (int a = 0; a < V; ++a) f[a] = m.w[a] * amp * rng.gauss();
            int E = 0;
            if (!collide_fx<SET, N, false>(m.consts(tau, dt, 0.0), tau, dt, f, out, E)) continue;
            collide_ref<N, Q>(m, tau, dt, 0.0, f, ref);
            for (int a = 0; a < V; ++a) {
                const double e = double(fabsl(Q(out[a]) - ref[a]) / Q(amp));
                if (!(e <= worst)) worst = e;
            }
        }
        std::printf("%s: worst error %.3g of the amplitude\n", name, worst);
        return worst < 1e-12 ? 0 : 1;
    });
    return bad ? 1 : 0;
}

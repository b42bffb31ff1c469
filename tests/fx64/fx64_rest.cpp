// A fluid at rest at unit density without a force stays exactly so: a node whose
// populations are all zero is left to the FP64 form or returns zeros for zeros.
#include "fx64_ref.h"

int main() {
    const int bad = every_set([&](const auto& m, auto set, const char* name) {
        using SET = decltype(set);
        constexpr int V = SET::R + 2 * SET::P, N = 3;
        int wrong = 0;
        std::vector<double> f(V, 0.0), out;
        int E = 0;
        for (double Kn : {0.1, 1.0, 100.0}) {
            const double tau = std::sqrt(2 / M_PI) * Kn, dt = 1 / (64 * m.c);
            if (collide_fx<SET, N, false>(m.consts(tau, dt, 0.0), tau, dt, f, out, E))
                for (double v : out) wrong |= v != 0.0;
        }
        if (wrong) std::printf("%s: zeros do not stay zero (%.3g)\n", name, out[0]);
        return wrong;
    });
    return bad ? 1 : 0;
}

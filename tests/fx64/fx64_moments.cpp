// Rounding of a node's density and momentum by the fixed-point collision: mean
// and rms of its error against long double over random channel states, in units
// U_G of the node, beside those of the same formulas in fp64.  A mean error acts on
// the flow like a source or a body force.  The rms is below that of fp64 (U_G is
// 2^-56 of the largest |e| d where an fp64 population has 2^-53); the mean, which
// ties and truncated low words leave, is within a quarter of the fp64 rms, or
// of the mean of fp64 where that is larger.
#include "fx64_ref.h"

int main() {
    const int nodes = 60000;
    const int bad = every_set([&](const auto& m, auto set, const char* name) {
        using SET = decltype(set);
        constexpr int V = SET::R + 2 * SET::P, N = SET::P == 16 && SET::R ? 4 : 3;
        struct { double Kn, Ny, ma, amp, um, ne; } cases[] = {{0.1, 64, 1e-3, 1e-3, 1e-3, 1e-4}, {0.01, 2000, 1e-3, 1e-6, 1e-3, 1e-5},
                                                              {1.0, 64, 1e-2, 1e-3, 1e-2, 1e-3}, {0.2, 200, 1e-3, 0.1, 1e-2, 1e-2}};
        int wrong = 0;
        for (const auto& q : cases) {
            Random rng(20151029);
            const double tau = std::sqrt(2 / M_PI) * q.Kn, dt = 1 / (q.Ny * m.c), g = 8 * tau * q.ma;
            const fx::Consts k = m.consts(tau, dt, g);
            int n = 0;
            double sum[3] = {}, sq[3] = {}, dsum[3] = {}, dq[3] = {};
            for (int t = 0; t < nodes; ++t) {
                std::vector<double> f(V), out, dp;
                std::vector<Q> ref;
                const double d = q.amp * rng.gauss(), X = m.c * q.um * rng.gauss(), Y = m.c * q.um * rng.gauss();
                for (int a = 0; a < V; ++a) f[a] = m.w[a] * (d + m.ex[a] * X + m.ey[a] * Y + q.ne * rng.gauss());
                int E = 0;
                if (!collide_fx<SET, N, true>(k, tau, dt, f, out, E)) continue;
                ++n;
                collide_ref<N, Q>(m, tau, dt, g, f, ref);
                collide_ref<N, double>(m, tau, dt, g, f, dp);
                Q e[3] = {}, h[3] = {};
                for (int a = 0; a < V; ++a) {
                    const Q v = Q(out[a]) - ref[a], u = Q(dp[a]) - ref[a];
                    e[0] += v; e[1] += v * m.ex[a]; e[2] += v * m.ey[a];
                    h[0] += u; h[1] += u * m.ex[a]; h[2] += u * m.ey[a];
                }
                for (int i = 0; i < 3; ++i) {
                    const double x = double(e[i] / unit_g<SET>(E)), y = double(h[i] / unit_g<SET>(E));
                    sum[i] += x; sq[i] += x * x; dsum[i] += y; dq[i] += y * y;
                }
            }
            std::printf("%s Kn %g:", name, q.Kn);
            for (int i = 0; i < 3; ++i) {
                const double mean = sum[i] / n, rms = std::sqrt(sq[i] / n), se = rms / std::sqrt(double(n));
                const double dmean = dsum[i] / n, drms = std::sqrt(dq[i] / n);
                std::printf("  %s %+.3f +- %.3f (fp64 %+.3f), rms %.2f (fp64 %.2f)", i == 0 ? "rho" : (i == 1 ? "jx" : "jy"), mean,
                            se, dmean, rms, drms);
                if (std::fabs(mean) > std::fmax(drms / 4, std::fabs(dmean)) + 5 * se || rms > drms) wrong = 1;
            }
            std::printf("\n");
            if (n < nodes * 9 / 10) wrong = 1;
        }
        return wrong;
    });
    return bad ? 1 : 0;
}

// Compares the fixed-point fp64 collision (csrc/fx64.cuh, host build) with a
// long-double evaluation of the same scheme on random nodes of every compiled
// velocity set.  argv: number of nodes per regime.  Prints one line per set,
// order, force and regime: nodes taken by the fixed-point form, nodes left to
// the general form, and the largest error in units of its bound.
//
// Bound on a population's error: half an ulp of the result and of the target T
// (d* = (1 - omega) d + T, T rounded to fp64 once) plus omega w B U_G with U_G = 2^(E - 1074 - S0) and B the rounding of the sums and coefficients:
// V/2 units from drho, c^2 m sum|e| / 2 from J (m the largest component), and
// two units for each coefficient times its power of e, 2 (1 + 2 m + 3 m^2 +
// 4 m^3 + 5 m^4) over all orders; the higher orders carry extra bits, so this
// holds with room.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>

#include "dvm_sets.h"
#include "fx64.cuh"

using namespace lbm;
typedef long double Q;

static std::mt19937_64 rng(20151029);
static double gauss() { static std::normal_distribution<double> n; return n(rng); }
static double unif(double a, double b) { return std::uniform_real_distribution<double>(a, b)(rng); }

// weights that make the set a quadrature are not needed: the collision is the
// same polynomial for any weights, so w falls off like the lattice Gaussian
template <class SET>
static void weights(double c, std::vector<double>& w) {
    const int V = SET::R + 2 * SET::P;
    w.assign(V, 0.0);
    double s = 0;
    for (int a = 0; a < V; ++a) {
        const int p = a < SET::R ? -1 : (a - SET::R) % SET::P;
        const double e2 = p < 0 ? 0 : SET::ex[p] * SET::ex[p] + SET::ey[p] * SET::ey[p];
        w[a] = std::exp(-0.5 * c * c * e2);
        s += w[a];
    }
    for (double& v : w) v /= s;
}

template <class SET, int N, bool FORCE>
static int run(const char* name, double c, int tries) {
    constexpr int V = SET::R + 2 * SET::P;
    std::vector<double> w;
    weights<SET>(c, w);
    std::vector<int> ex(V, 0), ey(V, 0);
    for (int a = SET::R; a < V; ++a) {
        const int p = (a - SET::R) % SET::P, s = a - SET::R < SET::P ? 1 : -1;
        ex[a] = s * SET::ex[p];
        ey[a] = s * SET::ey[p];
    }
    int bad = 0;
    // regimes: 0 channel-like, 1 any amplitude and noise, 2 single large populations
    for (int regime = 0; regime < 3; ++regime) {
        int taken = 0, left = 0;
        double worst = 0;
        for (int t = 0; t < tries; ++t) {
            const double Kn = std::pow(10.0, unif(-2, regime ? 1 : 0)), Ny = std::floor(unif(16, 2048));
            const double tau = std::sqrt(2 / M_PI) * Kn, dt = 1 / (Ny * c);
            const double g = FORCE ? (t % 2 ? -8 : 8) * tau * std::pow(10.0, unif(-4, regime ? -1 : -2)) : 0.0;
            const double omega = dt / (tau + 0.5 * dt), omo = 1 - omega;
            const fx::Consts k = fx::make_consts(c, tau, dt, g, SET::R, SET::P, ex.data(), ey.data(), w.data(),
                                                 fx::set_info<SET>());
            const double amp = regime ? std::pow(10.0, unif(-14, 0.5)) : 1e-3;
            const double um = regime ? std::pow(10.0, unif(-14, -0.5)) : 1e-3 * std::pow(10.0, unif(0, 1));
            const double ne = regime ? std::pow(10.0, unif(-14, 0.5)) : 1e-4;
            const double d0 = amp * gauss(), X = c * um * gauss(), Y = c * um * gauss();
            std::vector<double> f(V), fn(V);
            for (int a = 0; a < V; ++a) f[a] = w[a] * (d0 + ex[a] * X + ey[a] * Y + ne * gauss());
            if (regime == 2) f[rng() % V] *= std::pow(10.0, unif(0, 8));
            fx::Sums m;
            int E = 0;
            const bool ok = fx::collide<SET, N, FORCE>(
                k, omo, m, E, [&](int a, int, int, int) { return f[a]; },
                [&](int a, int, int, int, double v) { fn[a] = v; });
            if (!ok) { ++left; continue; }
            ++taken;
            Q d = 0, jx = 0, jy = 0, kxx = 0, kxy = 0, kyy = 0;
            for (int a = 0; a < V; ++a) {
                const Q v = f[a];
                d += v; jx += v * ex[a]; jy += v * ey[a];
                kxx += v * (ex[a] * ex[a]); kxy += v * (ex[a] * ey[a]); kyy += v * (ey[a] * ey[a]);
            }
            const Q C = c, rho = 1 + d, ux = C * jx / rho + (Q)dt * g / 2, uy = C * jy / rho, u2 = ux * ux + uy * uy;
            const Q kk = 1 / (2 * (Q)tau + dt), T2 = 2 * (Q)tau;
            const Q axx = (T2 * (C * C * kxx - d) + dt * rho * (ux * ux + T2 * g * ux)) * kk;
            const Q axy = (T2 * C * C * kxy + dt * rho * (ux * uy + (Q)tau * g * uy)) * kk;
            const Q ayy = (T2 * (C * C * kyy - d) + dt * rho * uy * uy) * kk;
            int mc = fx::set_emax<SET>();
            double se = 0;
            for (int a = 0; a < V; ++a) se += std::abs(ex[a]) + std::abs(ey[a]);
            const double B = V / 2.0 + c * c * mc * se / 2 +
                             2 * (1 + 2.0 * mc + 3.0 * mc * mc + 4.0 * mc * mc * mc + 5.0 * std::pow(mc, 4));
            const Q UG = ldexpl(1.0L, E - 1074 - fx::guard_bits<SET>());
            for (int a = 0; a < V; ++a) {
                const Q xx = C * ex[a], xy = C * ey[a], s = ux * xx + uy * xy;
                Q r = s + (s * s - u2) / 2;
                if (N >= 3) r += s * (s * s - 3 * u2) / 6;
                if (N >= 4) r += (s * s * (s * s - 6 * u2) + 3 * u2 * u2) / 24;
                Q F = rho * g * (xx + xx * s - ux);
                if (N >= 3)
                    F += (Q)g / 2 * (xx * (axx * (xx * xx - 1) + 2 * axy * xx * xy + ayy * (xy * xy - 1)) -
                                     2 * (axx * xx + axy * xy));
                const double omw = omega * w[a];
                const Q ref = (Q)omo * f[a] + (Q)omw * (d + rho * r + (Q)tau * F);
                const Q bound = ldexpl(fabsl(ref) + fabsl(ref - (Q)omo * f[a]), -53) + omw * (B * UG) + ldexpl(1.0L, -1070);
                const double e = double(fabsl((Q)fn[a] - ref) / bound);
                if (!(e <= worst)) worst = e;
            }
        }
        std::printf("%s N%d force %d regime %d: taken %d left %d worst %.3f\n", name, N, int(FORCE), regime, taken,
                    left, worst);
        if (!(worst <= 1.0) || (regime == 0 && left)) bad = 1;
    }
    return bad;
}

template <class SET, int N>
static int both(const char* name, double c, int tries) {
    return run<SET, N, true>(name, c, tries) + run<SET, N, false>(name, c, tries);
}

int main(int argc, char** argv) {
    const int n = argc > 1 ? std::atoi(argv[1]) : 2000;
    int bad = 0;
    bad += both<SetD2V16, 2>("D2V16", 0.86602540378443865, n) + both<SetD2V16, 3>("D2V16", 0.86602540378443865, n) +
           both<SetD2V16, 4>("D2V16", 0.86602540378443865, n);
    bad += both<SetD2V33, 3>("D2V33", 1.1587791906520175, n) + both<SetD2V33, 4>("D2V33", 1.1587791906520175, n);
    bad += both<SetD2V32, 3>("D2V32", 0.34040702226615838, n) + both<SetD2V32, 4>("D2V32", 0.34040702226615838, n);
    bad += both<SetD2V53, 3>("D2V53", 0.61910486274, n) + both<SetD2V53, 4>("D2V53", 0.61910486274, n);
    bad += both<SetD2V40, 3>("D2V40", 0.37787, n) + both<SetD2V48, 3>("D2V48", 0.40521, n);
    return bad ? 1 : 0;
}

// A node's collision in any floating-point type, and the compiled velocity sets
// with lattice speeds and weights, for the checks of csrc/fx64.cuh on the host.
#pragma once
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>

#include "dvm_sets.h"
#include "fx64.cuh"

using namespace lbm;
typedef long double Q;

// Velocities and weights of a set, planes in the solver's order.  The collision
// is the same polynomial for any weights, so w falls off like the lattice
// Gaussian instead of being a quadrature.
template <class SET>
struct Model {
    static constexpr int V = SET::R + 2 * SET::P;
    double c;
    std::vector<int> ex, ey;
    std::vector<double> w;
    explicit Model(double c_) : c(c_), ex(V, 0), ey(V, 0), w(V, 0.0) {
        double s = 0;
        for (int a = 0; a < V; ++a) {
            if (a >= SET::R) {
                const int p = (a - SET::R) % SET::P, sg = a - SET::R < SET::P ? 1 : -1;
                ex[a] = sg * SET::ex[p];
                ey[a] = sg * SET::ey[p];
            }
            w[a] = std::exp(-0.5 * c * c * (ex[a] * ex[a] + ey[a] * ey[a]));
            s += w[a];
        }
        for (double& v : w) v /= s;
    }
    fx::Consts consts(double tau, double dt, double g) const {
        return fx::make_consts(c, tau, dt, g, SET::R, SET::P, ex.data(), ey.data(), w.data(), fx::set_info<SET>());
    }
};

// d* of every population, in T, with the rounded 1 - omega and omega w of a solve.
template <int N, class T, class MODEL>
void collide_ref(const MODEL& m, double tau_, double dt_, double g_, const std::vector<double>& f, std::vector<T>& out) {
    const double omega = dt_ / (tau_ + 0.5 * dt_), omo = 1 - omega;
    const T c = m.c, tau = tau_, dt = dt_, g = g_;
    T d = 0, jx = 0, jy = 0, kxx = 0, kxy = 0, kyy = 0;
    for (int a = 0; a < MODEL::V; ++a) {
        const T v = f[a];
        d += v;
        jx += v * m.ex[a];
        jy += v * m.ey[a];
        kxx += v * (m.ex[a] * m.ex[a]);
        kxy += v * (m.ex[a] * m.ey[a]);
        kyy += v * (m.ey[a] * m.ey[a]);
    }
    const T rho = 1 + d, ux = c * jx / rho + dt * g / 2, uy = c * jy / rho, u2 = ux * ux + uy * uy;
    const T k = 1 / (2 * tau + dt), t2 = 2 * tau;
    const T axx = (t2 * (c * c * kxx - d) + dt * rho * (ux * ux + t2 * g * ux)) * k;
    const T axy = (t2 * c * c * kxy + dt * rho * (ux * uy + tau * g * uy)) * k;
    const T ayy = (t2 * (c * c * kyy - d) + dt * rho * uy * uy) * k;
    out.resize(MODEL::V);
    for (int a = 0; a < MODEL::V; ++a) {
        const T x = c * m.ex[a], y = c * m.ey[a], s = ux * x + uy * y;
        T r = s + (s * s - u2) / 2;
        if (N >= 3) r += s * (s * s - 3 * u2) / 6;
        if (N >= 4) r += (s * s * (s * s - 6 * u2) + 3 * u2 * u2) / 24;
        T F = rho * g * (x + x * s - ux);
        if (N >= 3) F += g / 2 * (x * (axx * (x * x - 1) + 2 * axy * x * y + ayy * (y * y - 1)) - 2 * (axx * x + axy * y));
        out[a] = T(omo) * T(f[a]) + T(omega * m.w[a]) * (d + rho * r + tau * F);
    }
}

// The fixed-point collision of f; false: left to the FP64 form.
template <class SET, int N, bool FORCE>
bool collide_fx(const fx::Consts& k, double tau, double dt, const std::vector<double>& f, std::vector<double>& out, int& E) {
    const double omega = dt / (tau + 0.5 * dt);
    fx::Sums s;
    out.assign(f.size(), 0.0);
    return fx::collide<SET, N, FORCE>(
        k, 1 - omega, s, E, [&](int a, int, int, int) { return f[a]; },
        [&](int a, int, int, int, double v) { out[a] = v; });
}

// unit of the target's coefficients
template <class SET>
Q unit_g(int E) { return ldexpl(1.0L, E - 1074 - fx::guard_bits<SET>()); }

struct Random {
    std::mt19937_64 r;
    std::normal_distribution<double> n;
    explicit Random(unsigned long long seed) : r(seed) {}
    double gauss() { return n(r); }
    double uniform(double a, double b) { return std::uniform_real_distribution<double>(a, b)(r); }
};

template <class FN>
int every_set(const FN& fn) {
    return fn(Model<SetD2V16>(0.86602540378443865), SetD2V16{}, "D2V16") +
           fn(Model<SetD2V33>(1.1587791906520175), SetD2V33{}, "D2V33") +
           fn(Model<SetD2V32>(0.34040702226615838), SetD2V32{}, "D2V32") +
           fn(Model<SetD2V53>(0.61910486274), SetD2V53{}, "D2V53") + fn(Model<SetD2V40>(0.37787), SetD2V40{}, "D2V40") +
           fn(Model<SetD2V48>(0.40521), SetD2V48{}, "D2V48");
}

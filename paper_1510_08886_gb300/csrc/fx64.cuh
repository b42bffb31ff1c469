// Collision of an fp64 node of a compiled velocity set on the integer pipes.
//
// GB300 has two FP64 lanes per SM: every warp-wide DADD, DMUL, DFMA and every
// conversion to or from fp64 holds its SMSP's FP64 unit for 64 cycles (measured),
// a 64-bit integer add takes 4, a 64 x 64 -> high 64 product about 17, a
// variable 64-bit shift 4.  The collision needs ~475 FP64 operations a node for
// the 33-velocity set, so the fp64 step ran at a tenth of the memory rate.
// Here everything between the load and the last fused multiply-add is 64-bit
// fixed point with one exponent per node:
//
//   in    every population d_a is rounded to a multiple of the node's unit
//         U = 2^(E - 1079) (S0 = 4 below), E the largest biased exponent of |e_a| d_a over the
//         populations (|e_a| rounded up to a power of two), so that no sum over
//         the populations can overflow and the unit lies 2^-55 below the largest
//         term;
//   sums  drho, J and K are exact integer sums;
//   out   the target of every population is formed with 64-bit products in the
//         unit U_G = 2 U, converted to fp64 (rounded to nearest) and relaxed
//         with one fma: d* = (1 - omega) d + omega w G.
//
// Roundings are to nearest but for ties and for the low words that a product or a
// shift drops, and a bias of a fraction of a unit per step acts on the flow like a
// body force: over random channel states (Kn 0.01 to 1, u 1e-3 to 1e-2, Ma to 1e-2)
// a node's mean error is up to 0.06 U_G in the density, 0.27 U_G in x and 0.09 U_G
// in y momentum, against 0.09, 2.2 and 0.15 in fp64 arithmetic.  The rms error is
// 0.17 to 0.78 of that of the same formulas in fp64 (tests/fx64/fx64_moments.cpp) and
// 0.2 to 1.2 of that of the FP64 form (dp_collide), which shares sums between the
// populations; in the first steps from rest, whose populations are far below the
// force's scale, density and y momentum, both near zero there, are at up to 2.
//
// Per 32 nodes and step (D2V33, N = 4) this issues 3707 instructions, 34 of them
// FP64, against ~475 FP64 ones of 64 cycles: 331 us per step on 4096 x 512 (1585 in
// FP64), D2V16 166 us (816), D2V53 2048 x 512 293 us (1044).
//
// Nodes outside the range of the fixed-point form (a density far from 1, a flow
// speed near the lattice's limit, non-finite values) and solves whose force
// constants do not fit take the FP64 evaluation (dp_collide), node by node.
//
// The functions are plain C++ with the device's multiply intrinsics spelled out
// for the host, so that the CPU tests run the same arithmetic.
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#include <utility>

#if defined(__CUDACC__)
#define LBM_HD __host__ __device__ __forceinline__
#define LBM_CX __host__ __device__ constexpr
#else
#define LBM_HD inline
#define LBM_CX constexpr
#endif

namespace lbm {
namespace fx {

using i64 = long long;
using u64 = unsigned long long;

// Multiplier m = h 2^32 + l with a signed low word, used as m 2^-64; r rounds
// the product: 1/2 unit plus the mean of the dropped product of the low words.
struct Mul {
    int h, l;
    unsigned r;
};
LBM_CX Mul make_mul(i64 n) {
    const int l = int(unsigned(n));
    return Mul{int((n - l) >> 32), l, 0x80000000u + unsigned(l / 2)};
}

// Populations with the same (|e_x|, |e_y|) = (ax, ay): planes a, am of e =
// (ax, ay) and -e, and off the axes b, bm of (-ax, ay) and its negative.
struct Row {
    int ax, ay;
    int a, am, b, bm;
    int lg;                  // log2 max(ax, ay), rounded up
    int oe;                  // omega w = om 2^-oe
    Mul om;
};
constexpr int kMaxRows = 32;

// Per-solve constants of the fixed-point collision; a trailing number is the
// constant's binary point: th_62 = theta 2^62.  With theta = tau c g and the
// momentum-flux deviation A of Eq. nm.4,
//   theta A_xx / 2 = k1 K_xx - k0 drho + k2 rho X^2 / 2 + k3 M_x, ...
struct Consts {
    int ok;                  // 1: the fixed-point form may be used
    int mirror;              // 1: g < 0, the constants are those of |g|
    int emin;                // least E: keeps h and theta in range
    int h_exp, th_exp;       // h = h_m 2^-h_exp, theta = th_m 2^-th_exp
    i64 h_m, th_m;           // 62-bit mantissas; h = c (dt/2) g
    Mul c2;                  // c^2, binary point c2_point(emax)
    Mul h_63, th_63;         // h, theta                      (times drho)
    Mul ic4_60;              // 1 / (4 c^2)
    Mul th_62_s2, thic_62;   // theta 2^s2, theta / c^2       (times M)
    Mul k1;                  // theta c^2 k / 2, k = 2 tau / (2 tau + dt); binary point 61 + kshift
    Mul k0_63;               // theta k / 2                   (times drho)
    Mul k2_60;               // theta dt / ((2 tau + dt) c^2) (times S / 2)
    Mul k3_62, k3h_62;       // theta tau g dt / ((2 tau + dt) c) and its half (times M)
    float gm, ga;            // bound on |G| and its partial sums from the high words of M and theta A
    float em;                // max |e|: the same from theta
    float xlim, c2f;         // bound on |X| + |Y|; c^2
    // rows [0, nx): e = (ax, 0); [nx, ny): (0, ay); [ny, nd): four velocities
    int nx, ny, nd, rest;    // rest: 1 if plane 0 is the rest population
    Mul om0;                 // omega w of the rest population = om0 2^-oe0
    int oe0, fam;            // fam: see FamilyFormat, -1: none fits
    Row row[kMaxRows];
    // per pair (plane order): omega w = pom 2^-poe
    Mul pom[kMaxRows];
    int poe[kMaxRows];
};

LBM_HD i64 mulw(int a, int b) { return i64(a) * b; }
LBM_HD i64 mulwu(unsigned a, unsigned b) { return i64(u64(a) * b); }

// x m 2^-64 + frac 2^-32, rounded to nearest, for 0 <= m < 2^62; three wide
// multiply-adds.
LBM_HD i64 mulc(i64 x, Mul m, unsigned frac = 0u) {
    const int xh = int(x >> 32);
    const unsigned xl = unsigned(x);
    const i64 mid = mulw(xh, m.l) + (i64(m.r) + i64(frac)) + mulwu(xl, unsigned(m.h));
    return mulw(xh, m.h) + (mid >> 32);
}

// The same for a variable multiplier of either sign, |m| < 2^62.
struct MulV {
    int h, l;
    unsigned s;              // all ones if h < 0
};
LBM_HD MulV mulv(i64 v) {
    MulV m;
    m.l = int(v);
    m.h = int(v >> 32) + (m.l < 0 ? 1 : 0);
    m.s = unsigned(m.h >> 31);
    return m;
}
LBM_HD i64 mulx(i64 x, const MulV& m) {
    const int xh = int(x >> 32);
    const unsigned xl = unsigned(x);
    // xl m.h with m.h taken modulo 2^32, 2^32 xl too much if m.h < 0
    const u64 mid = u64(mulw(xh, m.l)) + 0x80000000ull + u64(mulwu(xl, unsigned(m.h)));
    const int mh = int(unsigned(mid >> 32) - (xl & m.s));
    return mulw(xh, m.h) + i64(mh);
}

LBM_HD i64 shl(i64 x, int n) { return i64(u64(x) << n); }
// x 2^n for a constant n of either sign, rounded to nearest
LBM_HD i64 sh_(i64 x, int n) { return n >= 0 ? shl(x, n) : (x + (i64(1) << (-n - 1))) >> -n; }

LBM_HD int dhi(double d) {
#if defined(__CUDA_ARCH__)
    return __double2hiint(d);
#else
    i64 b; memcpy(&b, &d, 8); return int(b >> 32);
#endif
}
LBM_HD unsigned dlo(double d) {
#if defined(__CUDA_ARCH__)
    return unsigned(__double2loint(d));
#else
    i64 b; memcpy(&b, &d, 8); return unsigned(b);
#endif
}
LBM_HD double mkd(int hi, unsigned lo) {
#if defined(__CUDA_ARCH__)
    return __hiloint2double(hi, int(lo));
#else
    const u64 b = u64(unsigned(hi)) << 32 | lo; double d; memcpy(&d, &b, 8); return d;
#endif
}
LBM_HD int clz64(u64 x) {        // 64 for x = 0
#if defined(__CUDA_ARCH__)
    const unsigned h = unsigned(x >> 32), l = unsigned(x);
    return __clz(int(h ? h : l)) + (h ? 0 : 32);
#else
    return x ? __builtin_clzll(x) : 64;
#endif
}

// x >> sh for any sh >= 0 (the device's shift saturates at 63)
LBM_HD i64 asr(i64 x, int sh) {
#if defined(__CUDA_ARCH__)
    i64 y;
    asm("shr.s64 %0, %1, %2;" : "=l"(y) : "l"(x), "r"(sh));
    return y;
#else
    return x >> (sh < 63 ? sh : 63);
#endif
}

// Population d as a multiple of U = 2^(E - 1075 - S0), rounded to nearest, as an
// even integer.
template <int S0>
LBM_HD i64 to_fixed(double d, int E) {
    const int hi = dhi(d);
    const unsigned lo = dlo(d);
    const int sh = E - ((hi >> 20) & 0x7ff);           // 0 .. kLargestE
    const int s = hi >> 31;
    int xh = int((unsigned(hi) << S0) | (lo >> (32 - S0)));
    xh = ((xh & ((1 << (20 + S0)) - 1)) | (1 << (20 + S0))) ^ s;
    const unsigned xl = (lo << S0) ^ unsigned(s);
    const i64 x = i64(u64(unsigned(xh)) << 32 | xl);   // +- mantissa 2^S0 (one's complement)
    const i64 y = asr(x, sh);
    return i64(u64(y + 1) & ~u64(1));
}

// T 2^(eb - 1084) as a double, rounded to nearest; |T| < 2^62 (T = 0: a quarter of
// the unit).
LBM_HD double to_double(i64 T, int eb) {
    const int s = int(T >> 63);
    const u64 a = u64((T ^ i64(s)) - i64(s));
    const int n = clz64(a) - 1;                 // leading bit to bit 62
    const u64 x = ((a << n) + 0x200u) >> 10;    // bit 52 (or 53 after a carry)
    const int hi = int(unsigned(x >> 32) + unsigned((eb - n) << 20)) | (s & int(0x80000000u));
    return mkd(hi, unsigned(x));
}

// log2 of max(|ex|, |ey|, 1), rounded up
LBM_CX int ilog2_up(int v) {
    int n = 0;
    while ((1 << n) < v) ++n;
    return n;
}
template <class SET>
LBM_CX int comp_max(int p) {
    const int x = SET::ex[p] < 0 ? -SET::ex[p] : SET::ex[p], y = SET::ey[p] < 0 ? -SET::ey[p] : SET::ey[p];
    return x > y ? x : y;
}
template <class SET>
LBM_CX int set_emax() {
    int m = 0;
    for (int p = 0; p < SET::P; ++p) m = comp_max<SET>(p) > m ? comp_max<SET>(p) : m;
    return m;
}
// K is summed in units of 2^kshift U: sum e^2 |v| / 2^kshift <= sum e |v|
template <class SET>
LBM_CX int kshift() { return ilog2_up(set_emax<SET>()); }

// Bits kept below a population's last mantissa bit: e_a |d_a| 2^(S0 - E + 1075) is
// below 2^(53 + S0) e_a / k_a, k_a the power of two of the exponent key, so the
// sums stay below 2^63 for S0 = 5 if sum e_a / k_a <= 31, else for S0 = 4 (V < 64).
template <class SET>
LBM_CX int guard_bits() {
    if (set_emax<SET>() <= 8) return 4;
    int s = SET::R * 16;                       // 16 sum e_a / k_a
    for (int p = 0; p < SET::P; ++p) s += 2 * 16 * comp_max<SET>(p) / (1 << ilog2_up(comp_max<SET>(p)));
    return s <= 31 * 16 ? 5 : 4;
}

// Sets with long velocities have small lattice speeds (c^2 ~ 1 / e^2) and
// weigh the higher coefficients with e^2 and e^3: those carry more bits below
// U_G (s2 for the second and fourth order, s3 for the third), and c^2 < 1/2
// leaves room for a binary point of 63.
LBM_CX int c2_point(int emax) { return emax > 4 ? 63 : 61; }
LBM_CX int extra2(int emax) { return emax > 4 ? 2 : 0; }
LBM_CX int extra3(int emax) { return emax > 4 ? 5 : 0; }

// The binary points of a set's fixed-point form.
template <class SET>
struct Format {
    static constexpr int EMAX = set_emax<SET>(), S0 = guard_bits<SET>(), KS = kshift<SET>();
    static constexpr int S2 = extra2(EMAX), S3 = extra3(EMAX), C2 = c2_point(EMAX);
};
// The same for a kernel that knows only the number LP of lanes per node (pairs
// at most LP) and, for LP = 16, which of the two: 0 for components up to 4, 1 for
// up to 8, 2 above.  SetInfo::fam says which one fits a set.
template <int FAM>
struct FamilyFormat {
    static constexpr int EMAX = FAM == 0 ? 4 : (FAM == 1 ? 8 : 16), S0 = FAM == 2 ? 5 : 4, KS = ilog2_up(EMAX);
    static constexpr int S2 = extra2(EMAX), S3 = extra3(EMAX), C2 = c2_point(EMAX);
};

struct Sums {
    i64 d, jx, jy, kxx, kxy, kyy;
};

// Range of E.  Below: populations this small (2^-895) are those of a fluid at rest
// without a force, whose zeros the FP64 form keeps; to_double has none.
constexpr int kLeastE = 128, kLargestE = 1021;
LBM_HD bool exponent_fits(int E) { return E > kLeastE && E <= kLargestE; }

// Bits of the force's constants h and theta, times max |e|, in units U_G at most: the
// unit of a strong force is set by it, and fewer bits would round coarser than fp64.
constexpr int kForceRoom = 60;
// Binary exponent of h and theta below which const_q would shift by more than 63
// (q >= 1074 + 4 - kLargestE): solves with so small a force take the FP64 form.
constexpr int kLeastForce = 62 - 63 - (1074 + 4 - kLargestE);

// exponent key of |e| d, lg = log2 of |e|
LBM_HD unsigned key(double d, int lg) { return (unsigned(dhi(d)) & 0x7fffffffu) + (unsigned(lg) << 20); }
LBM_HD unsigned umax_(unsigned a, unsigned b) { return a > b ? a : b; }

// acc + k x for a small k >= 0 (one wide and one narrow multiply-add)
LBM_HD i64 madk(i64 acc, int k, i64 x) { return i64(u64(acc) + u64(unsigned(k)) * u64(x)); }

// Coefficients of the target polynomial in e (see PolyCoef): c00, d10, d01 in
// units U_G, the other c in units 2^-s2 U_G, the other d in units 2^-s3 U_G.
struct Poly {
    i64 c00, c20, c11, c02, c40, c31, c22, c13, c04;
    i64 d10, d01, d30, d21, d12, d03;
};

// x 2^-sh for sh of either sign, rounded down (|sh| < 64)
LBM_HD i64 scale2(i64 x, int sh) {
    const int r = sh > 0 ? (sh < 63 ? sh : 63) : 0, l = sh < 0 ? -sh : 0;
    return shl(x, l) >> r;
}

LBM_HD float hif(i64 x) { return float(int(x >> 32)); }   // x / 2^32
LBM_HD float fabsf_(float x) { return x < 0.f ? -x : x; }
LBM_HD float fmaxf_(float a, float b) { return a > b ? a : b; }
LBM_HD float exp2i(int n) {                               // 2^n, n in [-126, 127]
    const int b = (n + 127) << 23;
#if defined(__CUDA_ARCH__)
    return __int_as_float(b);
#else
    float f; memcpy(&f, &b, 4); return f;
#endif
}
LBM_HD float rcp_(float x) {
#if defined(__CUDA_ARCH__)
    return __frcp_rn(x);
#else
    return 1.0f / x;
#endif
}
LBM_HD int f2i(float x) {
#if defined(__CUDA_ARCH__)
    return __float2int_rn(x);
#else
    return int(lrintf(x));
#endif
}

// The per-solve constant mant 2^-exp in the unit 2^-q: integer part and the
// 32 bits below it.
LBM_HD i64 const_q(i64 mant, int exp, int q, unsigned& frac) {
    const int sh = exp - q;                                // 2 (emin) .. 63 (kLeastForce)
    frac = unsigned(u64(mant << (64 - sh)) >> 32);
    return mant >> sh;
}

constexpr float kGMax = 1.9e9f;      // of the high word of G: |G| < 2^62.9

// Target coefficients from the sums; false outside the fixed-point range.
// Binary points: U_G = 2^-q with q = 1074 + S0 - E; X, Y = c u and eps = drho / rho
// are multiples of 2^-62.  M = rho X, H = rho X X / 2, t = rho X X X / 2,
// a = rho X^4 / 4 (and the mixed products).  Shifts left before a product use
// the room the bounds leave, so that a product loses less than a unit.
template <class FMT, int N, bool FORCE>
LBM_HD bool coefs(const Consts& k, Sums m, int E, Poly& p) {
    // g < 0 is the mirror image in x of |g|: e_x -> -e_x before and after
    if (FORCE && k.mirror) {
        m.jx = -m.jx;
        m.kxy = -m.kxy;
    }
    constexpr int S2 = FMT::S2, S3 = FMT::S3, C2 = FMT::C2;
    const int q = 1074 + FMT::S0 - E;
    const float fd = hif(m.d), fj = fabsf_(hif(m.jx)) + fabsf_(hif(m.jy));
    float fk = 0.f;
    if (FORCE && N >= 3) fk = fabsf_(hif(m.kxx)) + fabsf_(hif(m.kxy)) + fabsf_(hif(m.kyy));
    const float un = exp2i(q < 150 ? 31 - q : -119);       // high word of a sum -> its value
    const float delta = fd * un;
    unsigned hfrac = 0u, tfrac = 0u;
    i64 hq = 0, tq = 0;
    // bounds on |M| (high word, and as a value: |X| + |Y|) and |G|
    float fm = 0.5f * k.c2f * fj, bound = fabsf_(fd);
    if (FORCE) {
        hq = const_q(k.h_m, k.h_exp, q, hfrac);
        tq = const_q(k.th_m, k.th_exp, q, tfrac);
        const float rho = 1.0f + delta;
        fm += rho * hif(hq);
        bound += rho * k.em * hif(tq);
    }
    bound += k.gm * fm;
    // left early: a node out of range pays for the sums only
    if (!(fj < (C2 == 61 ? 5.0e8f : 1.9e9f) && fk < 5.0e8f && 2.0f * fm * un < k.xlim && delta > -0.4f &&
          delta < 1.9f && bound < kGMax))
        return false;

    i64 Mx = mulc(shl(m.jx, 63 - C2), k.c2, hfrac);
    const i64 My = mulc(shl(m.jy, 63 - C2), k.c2);
    if (FORCE) Mx += hq + mulc(m.d, k.h_63);
    const i64 dG = m.d >> 1;                               // m.d is even
    const i64 Mx2 = shl(Mx, 2), My2 = shl(My, 2);
    i64 X, Y;
    {   // eps = drho / rho: an fp32 start and two correction steps
        const int sh = q - 61;
        const i64 d61 = scale2(dG, sh);
        const float r0 = rcp_(1.0f + delta);
        i64 eps = shl(i64(f2i(delta * r0 * 1073741824.0f)), 32);
        const int r29 = f2i(r0 * 536870912.0f);            // 2^29 / rho
        const MulV dm = mulv(d61);
#pragma unroll
        for (int it = 0; it < 2; ++it) {
            // residual drho - eps (1 + drho), times 1 / rho
            const i64 R = shl(shl(d61, 1) - eps - shl(mulx(shl(eps, 1), dm), 2), 3);
            eps += mulw(int(R >> 32), r29) + (mulwu(unsigned(R), unsigned(r29)) >> 32);
        }
        const MulV em = mulv(eps);
        // X = M / rho = M - M eps
        const i64 X0 = scale2(Mx, sh - 1), Y0 = scale2(My, sh - 1);
        X = X0 - mulx(shl(X0, 2), em);
        Y = Y0 - mulx(shl(Y0, 2), em);
    }
    const MulV xm = mulv(X), ym = mulv(Y);
    // H, S and a in units 2^-S2 U_G, t in units 2^-S3 U_G
    // (Sxy with the extra bits: 2 Y instead of a shift that M has no room for)
    const i64 Hxx = mulx(shl(Mx, 1 + S2), xm), Hyy = mulx(shl(My, 1 + S2), ym);
    const i64 Sxy = S2 ? mulx(shl(Mx, 1 + S2), mulv(shl(Y, 1))) : mulx(shl(Mx, 2), ym);
    p.c00 = dG - shl(mulc(shl(Hxx + Hyy, 5 - S2), k.ic4_60), 1);
    p.c20 = Hxx;
    p.c11 = Sxy;
    p.c02 = Hyy;
    p.d10 = Mx;
    p.d01 = My;
    if (FORCE) {
        p.c00 -= mulc(Mx2, k.thic_62);
        p.c20 += mulc(Mx2, k.th_62_s2);
        p.c11 += mulc(My2, k.th_62_s2);
        p.d10 += tq + mulc(m.d, k.th_63, tfrac);
    }
    if (N >= 3) {
        constexpr Mul third_62 = make_mul(0x1555555555555555ll);    // 2^62 / 3
        const i64 t30 = mulx(shl(Hxx, 2 + S3 - S2), xm), t21 = mulx(shl(Hxx, 2 + S3 - S2), ym);
        const i64 t12 = mulx(shl(Hyy, 2 + S3 - S2), xm), t03 = mulx(shl(Hyy, 2 + S3 - S2), ym);
        p.d10 -= mulc(sh_(t30 + t12, 6 - S3), k.ic4_60);
        p.d01 -= mulc(sh_(t21 + t03, 6 - S3), k.ic4_60);
        p.d30 = mulc(shl(t30, 2), third_62);
        p.d21 = t21;
        p.d12 = t12;
        p.d03 = mulc(shl(t03, 2), third_62);
        if (N >= 4) {
            const i64 a40 = mulx(sh_(t30, 1 + S2 - S3), xm), a31 = mulx(sh_(t30, 1 + S2 - S3), ym);
            const i64 a22 = mulx(sh_(t21, 1 + S2 - S3), ym), a13 = mulx(sh_(t12, 1 + S2 - S3), ym);
            const i64 a04 = mulx(sh_(t03, 1 + S2 - S3), ym);
            const i64 wx = mulc(shl(a40 + a22, 6), k.ic4_60), wy = mulc(shl(a22 + a04, 6), k.ic4_60);
            p.c00 += mulc(shl(wx + wy, 5 - S2), k.ic4_60);
            p.c20 -= wx;
            p.c11 -= mulc(shl(a31 + a13, 7), k.ic4_60);
            p.c02 -= wy;
            p.c40 = mulc(shl(a40, 1), third_62);
            p.c31 = mulc(shl(a31, 3), third_62);
            p.c22 = a22;
            p.c13 = mulc(shl(a13, 3), third_62);
            p.c04 = mulc(shl(a04, 1), third_62);
        }
        if (FORCE) {
            // theta A / 2, A = Pi - rho delta
            const i64 kd = mulc(m.d, k.k0_63);
            const i64 axx = mulc(shl(m.kxx, 2), k.k1) - kd + mulc(shl(Hxx, 4 - S2), k.k2_60) + mulc(Mx2, k.k3_62);
            const i64 axy = mulc(shl(m.kxy, 2), k.k1) + mulc(sh_(Sxy, 3 - S2), k.k2_60) + mulc(My2, k.k3h_62);
            const i64 ayy = mulc(shl(m.kyy, 2), k.k1) - kd + mulc(shl(Hyy, 4 - S2), k.k2_60);
            bound += k.ga * (fabsf_(hif(axx)) + fabsf_(hif(axy)) + fabsf_(hif(ayy)));
            p.d10 -= 3 * axx + ayy;
            p.d01 -= 2 * axy;
            p.d30 += mulc(shl(axx, 64 - C2 + S3), k.c2);
            p.d21 += mulc(shl(axy, 65 - C2 + S3), k.c2);
            p.d12 += mulc(shl(ayy, 64 - C2 + S3), k.c2);
        }
    }
    if (FORCE && k.mirror) {
        p.c11 = -p.c11;
        p.d10 = -p.d10;
        if (N >= 3) {
            p.d30 = -p.d30;
            p.d12 = -p.d12;
        }
        if (N >= 4) {
            p.c31 = -p.c31;
            p.c13 = -p.c13;
        }
    }
    return bound < kGMax;
}

// d* = (1 - omega) d + T, T = G omega w already scaled (units 2^(eb - 1084))
LBM_HD double relax(double omo, double f, i64 T, int eb) { return fma(omo, f, to_double(T, eb)); }

// Memory that get() reads is read again after this point: the populations need
// not stay in registers from one phase to the next.
LBM_HD void phase() {
#if defined(__CUDA_ARCH__)
    asm volatile("" ::: "memory");
#endif
}

// Row r of a set known at compile time (the rows of make_consts).
struct RowE {
    int ax, ay, a, am, b, bm, lg;
};
template <class SET>
struct Rows {
    int nx = 0, ny = 0, nd = 0;
    RowE row[kMaxRows] = {};
};
template <class SET>
LBM_CX Rows<SET> make_rows() {
    Rows<SET> t;
    for (int kind = 0; kind < 3; ++kind) {
        for (int p = 0; p < SET::P; ++p) {
            const int x = SET::ex[p], y = SET::ey[p];
            if (kind != (y == 0 ? 0 : (x == 0 ? 1 : 2)) || x < 0) continue;
            int q = p;
            if (kind == 2)
                for (int j = 0; j < SET::P; ++j)
                    if (SET::ex[j] == -x && SET::ey[j] == y) q = j;
            t.row[t.nd++] = RowE{x, y, SET::R + p, SET::R + SET::P + p, SET::R + q, SET::R + SET::P + q,
                                 ilog2_up(x > y ? x : y)};
        }
        if (kind == 0) t.nx = t.nd;
        if (kind <= 1) t.ny = t.nd;
    }
    return t;
}
template <class SET, int I>
struct CtRow {
    static constexpr Rows<SET> t = make_rows<SET>();
    static constexpr int ax = t.row[I].ax, ay = t.row[I].ay, a = t.row[I].a, am = t.row[I].am;
    static constexpr int b = t.row[I].b, bm = t.row[I].bm, lg = t.row[I].lg;
};

// body(row, per-solve row) for the rows [lo, hi): unrolled with the set's own
// numbers, or a loop over the solve's table.
template <class SET, int LO, class BODY, int... I>
LBM_HD void each_ct(const Consts& k, const BODY& body, std::integer_sequence<int, I...>) {
    (body(CtRow<SET, LO + I>{}, k.row[LO + I]), ...);
}
template <class SET, bool CT, int LO, int HI, class BODY>
LBM_HD void each_row(const Consts& k, const BODY& body) {
    if constexpr (CT) {
        each_ct<SET, LO>(k, body, std::make_integer_sequence<int, HI - LO>{});
    } else {
#pragma unroll 1
        for (int r = LO; r < HI; ++r) body(k.row[r], k.row[r]);
    }
}

// The collision of a node.  get(a, am, ex, ey): population a before the
// collision, of velocity (ex, ey), am the plane of the opposite velocity; called
// three times per population (exponents, sums, relaxation), so a read of shared
// memory.  put(a, am, ex, ey, v): its new value; a population and its opposite
// are read before either is put.  Returns false, nothing put, when the node is
// outside the fixed-point range.  m and E: the node's sums, for the moments a
// caller may want (value m.d 2^(E - 1075 - S0)).
template <class SET, int N, bool FORCE, class GET, class PUT>
LBM_HD bool collide(const Consts& k, double omo, Sums& m, int& E, const GET& get, const PUT& put) {
    constexpr int S0 = guard_bits<SET>(), EMAX = set_emax<SET>(), S2 = extra2(EMAX), S3 = extra3(EMAX);
    constexpr int KS = kshift<SET>();
    constexpr bool K = FORCE && N >= 3;
    constexpr Rows<SET> rows = make_rows<SET>();
    constexpr int NX = rows.nx, NY = rows.ny, ND = rows.nd;
    // Unrolled with the set's numbers, or loops over the solve's table: the
    // relaxation of sets of more than 16 pairs is a loop, its unrolled code
    // overruns the instruction caches (D2V53 2048 x 512, us per step: all
    // loops 314, all unrolled 324, only the relaxation a loop 303; D2V33
    // 4096 x 512: 357, 334, 339; D2V16: 191, 166, 179).
    constexpr bool UR = SET::P <= 16;
    if (!k.ok) return false;
    unsigned t = unsigned(k.emin) << 20;
    if constexpr (SET::R != 0) t = umax_(t, key(get(0, 0, 0, 0), 0));
    each_row<SET, true, 0, NY>(k, [&](const auto& w, const Row&) {
        t = umax_(t, umax_(key(get(w.a, w.am, w.ax, w.ay), w.lg), key(get(w.am, w.a, -w.ax, -w.ay), w.lg)));
    });
    each_row<SET, true, NY, ND>(k, [&](const auto& w, const Row&) {
        t = umax_(t, umax_(key(get(w.a, w.am, w.ax, w.ay), w.lg), key(get(w.am, w.a, -w.ax, -w.ay), w.lg)));
        t = umax_(t, umax_(key(get(w.b, w.bm, -w.ax, w.ay), w.lg), key(get(w.bm, w.b, w.ax, -w.ay), w.lg)));
    });
    E = int(t >> 20);
    if (!exponent_fits(E)) return false;
    phase();
    m = Sums{0, 0, 0, 0, 0, 0};
    if constexpr (SET::R != 0) m.d = to_fixed<S0>(get(0, 0, 0, 0), E);
    // K is summed in units of 2^KS U, rounded
    auto ku = [](i64 v) { return (v + (i64(1) << KS >> 1)) >> KS; };
    auto axis = [&](const auto& w, int e, i64& j, i64& kk) {
        const i64 vp = to_fixed<S0>(get(w.a, w.am, w.ax, w.ay), E);
        const i64 vm = to_fixed<S0>(get(w.am, w.a, -w.ax, -w.ay), E);
        m.d += vp + vm;
        j = madk(j, e, vp - vm);
        if constexpr (K) kk = madk(kk, e * e, ku(vp + vm));
    };
    each_row<SET, true, 0, NX>(k, [&](const auto& w, const Row&) { axis(w, w.ax, m.jx, m.kxx); });
    each_row<SET, true, NX, NY>(k, [&](const auto& w, const Row&) { axis(w, w.ay, m.jy, m.kyy); });
    each_row<SET, true, NY, ND>(k, [&](const auto& w, const Row&) {
        const i64 ap = to_fixed<S0>(get(w.a, w.am, w.ax, w.ay), E);
        const i64 am = to_fixed<S0>(get(w.am, w.a, -w.ax, -w.ay), E);
        const i64 bp = to_fixed<S0>(get(w.b, w.bm, -w.ax, w.ay), E);
        const i64 bm = to_fixed<S0>(get(w.bm, w.b, w.ax, -w.ay), E);
        const i64 sa = ap + am, sb = bp + bm, da = ap - am, db = bp - bm;
        m.d += sa + sb;
        m.jx = madk(m.jx, w.ax, da - db);
        m.jy = madk(m.jy, w.ay, da + db);
        if constexpr (K) {
            const i64 s = ku(sa + sb);
            m.kxx = madk(m.kxx, w.ax * w.ax, s);
            m.kyy = madk(m.kyy, w.ay * w.ay, s);
            m.kxy = madk(m.kxy, w.ax * w.ay, ku(sa - sb));
        }
    });
    Poly p;
    if (!coefs<Format<SET>, N, FORCE>(k, m, E, p)) return false;
    phase();
    // G = Ge +- Go of e and -e: Ge = Ee + sx sy Eo, Go = sx Ox + sy Oy with sx, sy
    // the signs of the components (see PolyCoef); T = G omega w
    const int eb = E + 10 + 64 - S0;                 // U_G = 2^(E - 1074 - S0)
    if constexpr (SET::R != 0) put(0, 0, 0, 0, relax(omo, get(0, 0, 0, 0), mulc(p.c00, k.om0), eb - k.oe0));
    auto axis_out = [&](const auto& w, const Row& o, int e, i64 c2, i64 c4, i64 d1, i64 d3) {
        const int e2 = e * e;
        i64 ev = madk(0, e2, c2), od = 0;
        if constexpr (N >= 4) ev = madk(ev, e2 * e2, c4);
        if constexpr (N >= 3) od = madk(0, e * e2, d3);
        const i64 Ge = mulc(p.c00 + sh_(ev, -S2), o.om), Go = mulc(madk(sh_(od, -S3), e, d1), o.om);
        const double fp = get(w.a, w.am, w.ax, w.ay), fm = get(w.am, w.a, -w.ax, -w.ay);
        put(w.a, w.am, w.ax, w.ay, relax(omo, fp, Ge + Go, eb - o.oe));
        put(w.am, w.a, -w.ax, -w.ay, relax(omo, fm, Ge - Go, eb - o.oe));
    };
    each_row<SET, UR, 0, NX>(k, [&](const auto& w, const Row& o) {
        axis_out(w, o, w.ax, p.c20, p.c40, p.d10, p.d30);
    });
    each_row<SET, UR, NX, NY>(k, [&](const auto& w, const Row& o) {
        axis_out(w, o, w.ay, p.c02, p.c04, p.d01, p.d03);
    });
    each_row<SET, UR, NY, ND>(k, [&](const auto& w, const Row& o) {
        const int x2 = w.ax * w.ax, y2 = w.ay * w.ay, xy = w.ax * w.ay;
        i64 ee = madk(madk(0, x2, p.c20), y2, p.c02), eo = madk(0, xy, p.c11), ox = 0, oy = 0;
        if constexpr (N >= 4) {
            ee = madk(madk(madk(ee, x2 * x2, p.c40), xy * xy, p.c22), y2 * y2, p.c04);
            eo = madk(madk(eo, xy * x2, p.c31), xy * y2, p.c13);
        }
        if constexpr (N >= 3) {
            ox = madk(madk(0, x2 * w.ax, p.d30), xy * w.ay, p.d12);
            oy = madk(madk(0, y2 * w.ay, p.d03), xy * w.ax, p.d21);
        }
        const i64 Ee = mulc(p.c00 + sh_(ee, -S2), o.om), Eo = mulc(sh_(eo, -S2), o.om);
        const i64 Ox = mulc(madk(sh_(ox, -S3), w.ax, p.d10), o.om);
        const i64 Oy = mulc(madk(sh_(oy, -S3), w.ay, p.d01), o.om);
        const int eh = eb - o.oe;
        {
            const double fp = get(w.a, w.am, w.ax, w.ay), fm = get(w.am, w.a, -w.ax, -w.ay);
            const i64 e = Ee + Eo, q = Ox + Oy;
            put(w.a, w.am, w.ax, w.ay, relax(omo, fp, e + q, eh));
            put(w.am, w.a, -w.ax, -w.ay, relax(omo, fm, e - q, eh));
        }
        {
            const double fp = get(w.b, w.bm, -w.ax, w.ay), fm = get(w.bm, w.b, w.ax, -w.ay);
            const i64 e = Ee - Eo, q = Oy - Ox;
            put(w.b, w.bm, -w.ax, w.ay, relax(omo, fp, e + q, eh));
            put(w.bm, w.b, w.ax, -w.ay, relax(omo, fm, e - q, eh));
        }
    });
    return true;
}

// Target of the pair of velocity (ex, ey), before the weight: Ge +- Go for the
// member and its negative (the polynomial in e evaluated for one pair).
template <class FMT, int N>
LBM_HD void pair_target(const Poly& p, int ex, int ey, i64& Ge, i64& Go) {
    const int x2 = ex * ex, y2 = ey * ey, xy = ex * ey;
    i64 ev = madk(madk(0, x2, p.c20), y2, p.c02) + i64(xy) * p.c11, od = 0;
    if (N >= 4) {
        ev = madk(madk(madk(ev, x2 * x2, p.c40), xy * xy, p.c22), y2 * y2, p.c04);
        ev += i64(xy * x2) * p.c31 + i64(xy * y2) * p.c13;
    }
    if (N >= 3)
        od = i64(x2 * ex) * p.d30 + i64(xy * ey) * p.d12 + i64(y2 * ey) * p.d03 + i64(xy * ex) * p.d21;
    Ge = p.c00 + sh_(ev, -FMT::S2);
    Go = i64(ex) * p.d10 + i64(ey) * p.d01 + sh_(od, -FMT::S3);
}

// What the constants need to know of a velocity set.
struct SetInfo {
    int emax, ks, s0, fam;
};
template <class SET>
LBM_CX SetInfo set_info() {
    using F = Format<SET>;
    const int fam = F::EMAX <= 4 ? 0 : (F::EMAX <= 8 ? 1 : 2);
    const bool fits = fam == 0 ? F::S0 == FamilyFormat<0>::S0 && F::KS == FamilyFormat<0>::KS
                     : fam == 1 ? F::S0 == FamilyFormat<1>::S0 && F::KS == FamilyFormat<1>::KS
                                : F::S0 == FamilyFormat<2>::S0 && F::KS == FamilyFormat<2>::KS;
    return SetInfo{F::EMAX, F::KS, F::S0, fits ? fam : -1};
}

// Host: the constants of a solve (lattice speed c, relaxation time tau, time
// step dt, force g along x) of a set with planes e = (ex, ey), weights w, the
// rest plane first if R = 1, then P pair members and their negatives.  ok = 0 if
// a constant leaves its range (very large forces or Knudsen numbers).
inline Mul to_mul(long double v, int point, int& ok) {
    const long double x = ldexpl(v, point);
    if (!(x >= 0.0L && x < 4611686018427387904.0L)) { ok = 0; return Mul{0, 0, 0}; }
    return make_mul(i64(rintl(x)));
}

// omega w = m 2^-oe with m in [2^61, 2^62).  A target's biased exponent is at least
// E + 69 - oe - 62 (relax): oe may not exceed the least E by more than 6.
inline Mul to_weight(double ow, int& oe, int& ok) {
    int e = 0;
    frexp(ow, &e);
    oe = 62 - e;
    if (oe > kLeastE + 7) ok = 0;
    return to_mul(ow, oe, ok);
}

inline Consts make_consts(double c_, double tau_, double dt_, double g_, int R, int P, const int* ex,
                          const int* ey, const double* w, const SetInfo& si) {
    const int emax = si.emax, ks = si.ks;
    Consts k;
    memset(&k, 0, sizeof(k));
    if (emax < 1) return k;
    const long double c = c_, tau = tau_, dt = dt_, g = fabs(g_);
    k.mirror = g_ < 0.0;
    const long double h = 0.5L * dt * g * c, th = tau * c * g, k2t = 1.0L / (2 * tau + dt);
    k.ok = 1;
    k.emin = kLeastE;
    for (int i = 0; i < 2; ++i) {
        const long double v = i ? th : h;
        int e = 0;
        i64 mant = 0;
        if (v > 0) {
            mant = i64(ldexpl(frexpl(v, &e), 62));          // v = mant 2^(e - 62)
            // v 2^q < 2^room with q = 1074 + s0 - E
            const int room = kForceRoom - ilog2_up(emax);
            if (1074 + si.s0 + e - room > k.emin) k.emin = 1074 + si.s0 + e - room;
            if (e < kLeastForce) k.ok = 0;
        }
        (i ? k.th_m : k.h_m) = mant;
        (i ? k.th_exp : k.h_exp) = 62 - e;
    }
    // the rounding of the sums K enters the odd coefficients times theta c^4 e^3:
    // below that of fp64 for theta < 1/8 (8 tau^2 c Ma: Kn up to 4 at Ma = 1e-3)
    if (k.emin > kLargestE || th >= 0.125L) k.ok = 0;
    k.c2 = to_mul(c * c, c2_point(emax), k.ok);
    k.h_63 = to_mul(h, 63, k.ok);
    k.th_63 = to_mul(th, 63, k.ok);
    k.ic4_60 = to_mul(0.25L / (c * c), 60, k.ok);
    k.th_62_s2 = to_mul(th, 62 + extra2(emax), k.ok);
    k.thic_62 = to_mul(th / (c * c), 62, k.ok);
    k.k1 = to_mul(0.5L * th * c * c * 2 * tau * k2t, 61 + ks, k.ok);
    k.k0_63 = to_mul(0.5L * th * 2 * tau * k2t, 63, k.ok);
    k.k2_60 = to_mul(th * dt * k2t / (c * c), 60, k.ok);
    k.k3_62 = to_mul(th * tau * g * dt * k2t / c, 62, k.ok);
    k.k3h_62 = to_mul(0.5L * th * tau * g * dt * k2t / c, 62, k.ok);
    // M.e stays below 0.4 (xlim; the force's part h rho counts), so |G| < |drho| +
    // 1.3 M.e + theta rho e_x + ..., the sums of second order stay below 0.25 M.e and
    // those of third order below 0.04 M.e (in units with extra bits), besides the
    // theta M e^2 and theta A e^3 terms
    const float em = float(emax), f2 = float(1 << extra2(emax)), f3 = float(1 << extra3(emax));
    const float te = 2.0f * float(th) * em;
    float gj = 1.35f + te;
    if (f2 * (0.25f + te) > gj) gj = f2 * (0.25f + te);
    if (f3 * 0.05f > gj) gj = f3 * 0.05f;
    k.xlim = 0.4f / em;
    k.c2f = float(c * c);
    // M is shifted left by 3 bits with the extra bits, by 2 without, before a product:
    // |M| < 2^60 or 2^61 (a uniform flow's is at most 2^58.8 U_G in the paper's sets)
    const float room = extra2(emax) ? 2.4e8f : 4.8e8f;
    k.gm = em * gj > kGMax / room ? em * gj : kGMax / room;
    k.em = em;
    k.ga = f3 * (4.0f + 4.0f * k.c2f * em * em) * em;
    const double omega = dt_ / (tau_ + 0.5 * dt_);
    k.rest = R;
    k.fam = si.fam;
    if (P > kMaxRows) k.ok = 0;
    for (int p = 0; p < P && k.ok; ++p) k.pom[p] = to_weight(omega * w[R + p], k.poe[p], k.ok);
    if (R) k.om0 = to_weight(omega * w[0], k.oe0, k.ok);
    for (int kind = 0; kind < 3; ++kind) {
        for (int p = 0; p < P && k.ok; ++p) {
            const int a = R + p, x = ex[a], y = ey[a];
            // pair members have e_y > 0, or e_y = 0 and e_x > 0
            if (kind != (y == 0 ? 0 : (x == 0 ? 1 : 2)) || x < 0) continue;
            if (k.nd == kMaxRows) { k.ok = 0; break; }
            Row& r = k.row[k.nd++];
            r.ax = x;
            r.ay = y;
            r.a = a;
            r.am = a + P;
            r.lg = ilog2_up(x > y ? x : y);
            r.om = to_weight(omega * w[a], r.oe, k.ok);
            if (kind < 2) continue;
            int b = -1;
            for (int q = R; q < R + P; ++q)
                if (ex[q] == -x && ey[q] == y && fabs(w[q] - w[a]) <= 1e-15 * w[a]) b = q;
            if (b < 0) k.ok = 0;
            r.b = b;
            r.bm = b + P;
        }
        if (kind == 0) k.nx = k.nd;
        if (kind <= 1) k.ny = k.nd;
    }
    if (R + 2 * (k.ny + 2 * (k.nd - k.ny)) != R + 2 * P) k.ok = 0;
    return k;
}

}  // namespace fx
}  // namespace lbm

// lbm13_coef.h -- the per-lattice constants of the step: those of the
// collision (Coef, in lbm13_math.cuh) from the free parameters, the derived
// constants of Sec. 2 (lbm13_derive's output) and the boundary's force and
// energy source, and the wall arguments of the four sides (WallArgs, in
// lbm13_internal.h) with the correction polynomials of Sec. 7's walls.  Host
// code, used by lbm13_create.
#pragma once

#include <algorithm>

#include "lbm13_fixed_io.cuh"
#include "lbm13_internal.h"

namespace lbm13 {

// The constants of the integer collision (lbm13_fixed.cuh) from those of the
// FP64 one.  It is left off (on = 0) unless every coefficient is below 1 and the
// largest value that any sum can take at populations below 2^-5 stays inside 63
// bits; the parameter sets of params.py all pass.
// The sums of products behind each coefficient are taken in long double: their
// rounding in double would be the collision's largest error.
inline void fixed_coef(const lbm13_params &p, const double *D, const lbm13_boundary &b, const Coef<double> &k,
                       FixCoef<double> &x)
{
    using real = long double;
    x = FixCoef<double>{};
    bool ok = true;
    const auto to57 = [](real c) { return int64_t(std::llrint(std::ldexp(c, 57))); };
    const auto limb = [&](real c) {
        if (std::fabs(c) < real(1)) return fx_coef(to57(c));
        ok = false;
        return Limb{0, 0};
    };
    const real ME[4] = {-28, -15, -2, 24}, Meps[4] = {140, -2, -67, 34}, Mvpi[4] = {-12, 8, -6, 1};
    const double *rate = D + 9;
    const real lq = real(rate[6]) / 20, lr = real(rate[8]) / 70, lXX = real(rate[10]) / 68,
               lXXe = real(rate[12]) / 68, top = real(1) / 32;
    // scalar block: shells 0 and 1 per unit of shell sum and of the source (Coef::B, Coef::src)
    const real le = real(rate[2]) / 42196, lv = real(rate[3]) / 548;
    real B[2][4], s[2];
    for (int sh = 0; sh < 2; ++sh) {
        for (int l = 0; l < 4; ++l)
            B[sh][l] = Meps[sh] * le * (real(D[6]) + real(p.c_epsE) * ME[l] - Meps[l]) +
                       Mvpi[sh] * lv * (real(p.c_vpi_rho) + real(p.c_vpi_E) * ME[l] - Mvpi[l]);
        s[sh] = 13 * (Meps[sh] * le * real(p.c_epsE) + Mvpi[sh] * lv * real(p.c_vpi_E));
    }
    real r1[4], r9[4];
    for (int l = 0; l < 4; ++l) {
        x.B0[l] = limb(B[0][l]);
        x.B1[l] = limb(B[1][l]);
        // Q1 = Qh + h1 drho + k1 dE and R1 likewise, as sums over the shells
        const real dQ = real(k.h1) + real(k.k1) * ME[l], dR = real(k.h2) + real(k.k2) * ME[l];
        const real c1 = 4 * lr * dR - 2 * lq * dQ, c9 = 2 * lq * dQ + lr * dR;
        x.bA1[l] = limb(c1 / 8);
        x.bA9[l] = limb(c9 / 8);
        r1[l] = std::fabs(c1) * top;
        r9[l] = std::fabs(c9) * top;
    }
    const real E = real(p.E0) + 13 * real(b.heat);
    const real Qh = real(p.c1) + real(D[2]) + real(D[3]) * E, Rh = real(D[5]) + real(D[4]) + real(p.k2) * E;
    const real A10 = 4 * lr * Rh - 2 * lq * Qh, A90 = 2 * lq * Qh + lr * Rh;
    const real A1 = std::fabs(A10) + r1[0] + 4 * (r1[1] + r1[2] + r1[3]);
    const real A9 = std::fabs(A90) + r9[0] + 4 * (r9[1] + r9[2] + r9[3]);
    ok = ok && A1 < 2 && A9 < 2;
    x.A10 = ok ? to57(A10) : 0;
    x.A90 = ok ? to57(A90) : 0;
    // odd block: q = -2 b1 - dm + 2 b9, r = 4 b1 - 3 dm + b9
    const real c1[3] = {-16 * lr - 4 * lq, 12 * lr - 2 * lq, 4 * lq - 4 * lr};
    const real c9[3] = {4 * lq - 4 * lr, 2 * lq + 3 * lr, -4 * lq - lr};
    for (int i = 0; i < 3; ++i) {
        x.o1[i] = limb(c1[i]);
        x.o9[i] = limb(c9[i]);
    }
    // tensor block
    const real t11 = -lXX - 16 * lXXe, t19 = -4 * lXX + 4 * lXXe, t99 = -16 * lXX - lXXe;
    x.t11 = limb(t11);
    x.t19 = limb(t19);
    x.t99 = limb(t99);
    x.nXY = limb(-17 * lXX);
    ok = ok && lXX > 0 && lXX < real(1) / 32 && std::fabs(k.l_XY - 17.0 * k.l_XX) <= 1e-15;
    const int64_t l61 = ok ? to57(16 * lXX) : 0;
    x.lXXh = int(l61 >> 29);
    x.lXXl = int(l61 & ((1ll << 29) - 1));
    // force and source
    x.gx = limb(k.gx);
    x.gy = limb(k.gy);
    x.c14 = limb(real(1) / 14);
    x.c7 = limb(real(1) / 7);
    x.s0 = limb(s[0]);
    x.s1 = limb(s[1]);
    x.sE = limb(real(26) / 4004);
    x.cEF = limb(ok ? real(26) / 4004 / lXX : 0);
    x.Fx0 = (1.0 - k.rho_ref) * k.gx;
    x.Fy0 = (1.0 - k.rho_ref) * k.gy;
    x.q = b.heat;
    x.source = b.heat != 0.0;
    x.top = fx_mag(std::max({std::fabs(x.Fx0), std::fabs(x.Fy0), std::fabs(x.q)}));
    // with that, |F| is below 1.2 and |j + F/2| below 10.6 of the node's unit
    ok = ok && std::fabs(k.gx) < 1.0 / 64 && std::fabs(k.gy) < 1.0 / 64;
    // limb products of the odd block's sums inside 63 bits
    ok = ok && std::fabs(c1[0]) + std::fabs(c1[1]) + std::fabs(c1[2]) + A1 < real(5.5) &&
         std::fabs(c9[0]) + std::fabs(c9[1]) + std::fabs(c9[2]) + A9 < real(5.5);
    // Largest results in units of the largest population (2^59 of 2^63).  P (A -
    // A(rest)): a pair of opposite links gives to P what it does not give to the
    // shell sums, so that with fractions t the product is (sum p t)(r0 + sum r
    // (1 - t)) <= (c x + y / c)^2 / 4 for every c, and c x + y / c is largest
    // with each t at 0 or 1.
    const auto product = [](const real *r) {
        const real pr[6][2] = {{2, r[1]}, {0, r[1]}, {2, r[2]}, {2, r[2]}, {4, r[3]}, {0, r[3]}};
        real best = 1e30L;
        for (real c = 0.015625L; c < 4; c *= 1.05L) {
            real v = r[0] / c;
            for (const auto &e : pr) v += std::max(c * e[0], 2 * e[1] / c);
            best = std::min(best, v * v / 4);
        }
        return best;
    };
    // the linear part: row sums of its matrix, from the FP64 collision of small
    // single populations
    real row[Q] = {};
    for (int j = 0; j < Q; ++j) {
        double f[Q] = {};
        f[j] = 1e-9;
        collide_plain<false>(f, k);
        // the rest population may be 2^kFixRest times as large as the others, and
        // what it keeps of itself is not in the integers
        for (int i = 0; i < Q; ++i)
            row[i] += j > 0 ? std::fabs(f[i]) * real(1e9) : i > 0 ? std::fabs(f[i]) * real(1e9) * (1 << kFixRest) : 0;
    }
    // momentum flux at |j| < 10.6 / 32, rho > 0.59; the work of F and the source
    const real flux = lXX * real(10.6 * 10.6 / 0.59 / 32), p1 = product(r1) + real(0.6) * A1 + real(0.1),
               p9 = product(r9) + real(0.6) * A9 + real(0.2), dE = real(0.1), s0 = std::fabs(s[0]),
               s1 = std::fabs(s[1]);
    const real extra[4] = {28 * dE + s0, 15 * dE + s1 + p1 + flux, 2 * dE + s0 / 2 + 2 * s1 + p1 + 2 * p9 + 17 * flux,
                           24 * dE + s0 / 4 + s1 / 2 + p9 + 4 * flux};
    for (int j = 1; j < Q; ++j) ok = ok && row[j] + extra[j < 5 ? 1 : j < 9 ? 2 : 3] < real(15.9);
    // the scalar block's increment of the rest population, and what shells 9 and 5
    // are rounded from; with t > 0 the force's part is below 4 units too
    real in0 = 4 + s0, in9 = 0, in5 = 0;
    for (int l = 0; l < 4; ++l) {
        const real w = l == 0 ? 1 << kFixRest : 4;
        in0 += w * std::fabs(B[0][l]);
        in9 += w * std::fabs(B[0][l] + 2 * B[1][l]);
        in5 += w * std::fabs(B[0][l] + 3 * B[1][l]);
    }
    ok = ok && in0 < real(15.9) && in9 < real(15.9) && in5 < real(15.9);
    x.on = ok ? 1 : 0;
}

// D: the LBM13_DERIVED_COUNT constants of lbm13_derive (A, B, h1, k1, h2, c2,
// c_erho, sigma_XX, sigma_q, the 13 rates s_k, ...).
template <typename C>
void collision_coef(const lbm13_params &p, const double *D, const lbm13_boundary &b, Coef<C> &k)
{
    k.E0 = C(p.E0);
    k.cer = C(D[6]);
    k.ceE = C(p.c_epsE);
    k.cwr = C(p.c_vpi_rho);
    k.cwE = C(p.c_vpi_E);
    k.h1 = C(D[2]);
    k.k1 = C(D[3]);
    k.Q10 = C(p.c1 + D[2] + D[3] * p.E0);
    k.h2 = C(D[4]);
    k.k2 = C(p.k2);
    k.R10 = C(D[5] + D[4] + p.k2 * p.E0);
    const double *s = D + 9;
    k.l_eps = C(s[2] / kD[2]);
    k.l_vpi = C(s[3] / kD[3]);
    k.l_q = C(s[6] / kD[6]);
    k.l_r = C(s[8] / kD[8]);
    k.l_XX = C(s[10] / kD[10]);
    k.l_XY = C(s[11] / kD[11]);
    k.l_XXe = C(s[12] / kD[12]);
    k.gx = C(b.gx);
    k.gy = C(b.gy);
    k.rho_ref = C(b.rho_ref);
    // Energy source q (Sec. 9): equilibria at E + 13 q, so q_eq and r_eq
    // shift by 13 q k1 and 13 q k2 per unit of j.
    const double q = b.heat;
    k.Qh = q == 0.0 ? k.Q10 : C(p.c1 + D[2] + D[3] * (p.E0 + 13.0 * q));
    k.Rh = q == 0.0 ? k.R10 : C(D[5] + D[4] + p.k2 * (p.E0 + 13.0 * q));
    // Scalar block: values of the E, eps, varpi polynomials on the shells
    // (rest, unit axes, diagonals, distance-2 axes); the increment of a
    // population of shell s is eps_s d_eps + varpi_s d_varpi with
    // d_eps = l_eps (c_erho rho + c_epsE E - eps), all linear in the shell sums.
    const double ME[4] = {-28, -15, -2, 24}, Meps[4] = {140, -2, -67, 34}, Mvpi[4] = {-12, 8, -6, 1};
    const double le = s[2] / kD[2], lv = s[3] / kD[3];
    for (int sh = 0; sh < 4; ++sh)
        for (int l = 0; l < 4; ++l)
            k.B[sh][l] = C(Meps[sh] * le * (D[6] + p.c_epsE * ME[l] - Meps[l]) +
                           Mvpi[sh] * lv * (p.c_vpi_rho + p.c_vpi_E * ME[l] - Mvpi[l]));
    // Source: E* gains 26 q, eps and varpi relax toward equilibria raised by
    // 13 q c_epsE and 13 q c_varpiE.
    for (int sh = 0; sh < 4; ++sh)
        k.src[sh] = C(q == 0.0 ? 0.0
                               : ME[sh] * 26.0 * q / kD[1] + Meps[sh] * le * p.c_epsE * 13.0 * q +
                                     Mvpi[sh] * lv * p.c_vpi_E * 13.0 * q);
    // Tensor block: XX = X1 + 4 X9, XXe = -4 X1 + X9 relaxed and mapped back.
    const double lXX = s[10] / kD[10], lXXe = s[12] / kD[12];
    k.t1X1 = C(-lXX - 16.0 * lXXe);
    k.t1X9 = C(-4.0 * lXX + 4.0 * lXXe);
    k.t9X1 = C(-4.0 * lXX + 4.0 * lXXe);
    k.t9X9 = C(-16.0 * lXX - lXXe);
    if constexpr (sizeof(C) == sizeof(double)) fixed_coef(p, D, b, k, k.fx);
}

// The constants of the read-outs and of the initial state in integers
// (lbm13_fixed_io.cuh); off (on = 0) where a coefficient does not fit.
inline void read_fix(double E0, const lbm13_boundary &b, ReadFix &x)
{
    x = ReadFix{};
    const double T0 = (E0 + 28.0) / 26.0;
    if (!(T0 > 0.0 && T0 < 1.0 && std::fabs(b.gx) < 1.0 && std::fabs(b.gy) < 1.0)) return;
    const auto limb = [](double c) { return fx_coef(int64_t(std::llrint(std::ldexp(c, 57)))); };
    x.on = 1;
    x.T0 = limb(T0);
    const auto scaled = [&](double c, int &e) {
        std::frexp(c, &e);  // |c| < 2^e
        e = c == 0.0 ? 0 : std::min(std::max(-1 - e, 0), 60);
        return limb(std::ldexp(c, e));
    };
    x.hgx = scaled(0.5 * b.gx, x.ex);
    x.hgy = scaled(0.5 * b.gy, x.ey);
    x.Fx0 = 0.5 * (1.0 - b.rho_ref) * b.gx;
    x.Fy0 = 0.5 * (1.0 - b.rho_ref) * b.gy;
    x.half_q = 0.5 * b.heat;
}

inline void init_fix(const lbm13_params &p, const double *D, InitFix &x)
{
    using real = long double;
    x = InitFix{};
    bool ok = true;
    const auto limb = [&](real c) {
        if (std::fabs(c) < real(4)) return fx_coef(int64_t(std::llrint(std::ldexp(c, 57))));
        ok = false;
        return Limb{0, 0};
    };
    x.T0 = (p.E0 + 28.0) / 26.0;
    const real rest = 26 * real(x.T0) - 28;
    x.c0 = double((rest - real(p.E0)) / 16);
    x.rest = double(rest);
    x.dE0 = double(rest - real(p.E0));
    // dE / 16 = (26 rho dT + (26 T0 - 28) drho + 13 rho |u|^2) / 16 + c0
    x.z = limb(real(26) / 16);
    x.r = limb(rest / 16);
    x.k2 = limb(real(13) / 16);
    const real ME[4] = {-28, -15, -2, 24}, Meps[4] = {140, -2, -67, 34}, Mvpi[4] = {-12, 8, -6, 1};
    real top = 0;
    for (int s = 0; s < 4; ++s) {
        const real R = real(1) / 13 + Meps[s] * real(D[6]) / 42196 + Mvpi[s] * real(p.c_vpi_rho) / 548;
        const real E = ME[s] / 4004 + Meps[s] * real(p.c_epsE) / 42196 + Mvpi[s] * real(p.c_vpi_E) / 548;
        x.eR[s] = limb(R);
        x.eE[s] = limb(16 * E);
        x.R[s] = double(R);
        x.E[s] = double(E);
        top = std::max(top, std::fabs(R) + std::fabs(16 * E) * 4);
    }
    // unit and distance-2 links per unit of momentum: 1/14 - Q/10 + 2 R/35, 1/7 + Q/10 + R/70
    const real h1 = D[2], k1 = D[3], h2 = D[4], k2 = p.k2;
    const real Q0 = real(p.c1) + h1 + k1 * real(p.E0), R0 = real(D[5]) + h2 + k2 * real(p.E0);
    const real A10 = real(1) / 14 - Q0 / 10 + 2 * R0 / 35, A90 = real(1) / 7 + Q0 / 10 + R0 / 70;
    const real a1R = -h1 / 10 + 2 * h2 / 35, a1E = 16 * (-k1 / 10 + 2 * k2 / 35), a9R = h1 / 10 + h2 / 70,
               a9E = 16 * (k1 / 10 + k2 / 70);
    x.d10 = double(A10);
    x.l10 = double(A10 - real(x.d10));
    x.d1R = double(a1R);
    x.d1E = double(a1E / 16);
    x.d90 = double(A90);
    x.l90 = double(A90 - real(x.d90));
    x.d9R = double(a9R);
    x.d9E = double(a9E / 16);
    x.a1R = limb(a1R);
    x.a1E = limb(a1E);
    x.a9R = limb(a9R);
    x.a9E = limb(a9E);
    x.c68 = limb(real(1) / 68);
    // at deviations below 1/8, |dE| / 16 < 4 of them: A1 and A9 below 4 and every
    // sum below 2^62 (64 units of the largest deviation would be 2^63)
    const real A1 = std::fabs(A10) + (std::fabs(a1R) + 4 * std::fabs(a1E)) / 8;
    const real A9 = std::fabs(A90) + (std::fabs(a9R) + 4 * std::fabs(a9E)) / 8;
    ok = ok && A1 < 4 && A9 < 4 && std::fabs(rest) < 24 && top + 2 * (A1 + 2 * A9 + 1) + 1 < 30;
    x.A10 = ok ? int64_t(std::llrint(std::ldexp(A10, 57))) : 0;
    x.A90 = ok ? int64_t(std::llrint(std::ldexp(A90, 57))) : 0;
    x.on = ok ? 1 : 0;
}

// Coefficients (a0 .. a4) of P(drho, dE) = a0 + a1 drho + a2 dE + a3 drho^2 +
// a4 drho dE from values of P, which is exactly of that form: every
// equilibrium moment at rho = 1 + drho, E = E0 + dE, j = rho u is a
// combination of rho, E, rho^2 and rho E (Eq. d2q13-moments-equil).  The
// sample points rho = 1, 1 +- 1/2 and E0, E0 +- 1/2 give the coefficients
// without truncation error.
template <typename F>
void quadratic_coefficients(F P, double a[5])
{
    const double h = 0.5;
    const double p00 = P(0.0, 0.0), pp0 = P(h, 0.0), pm0 = P(-h, 0.0);
    const double p0p = P(0.0, h), p0m = P(0.0, -h), ppp = P(h, h);
    a[0] = p00;
    a[1] = (pp0 - pm0) / (2.0 * h);
    a[2] = (p0p - p0m) / (2.0 * h);
    a[3] = (pp0 + pm0 - 2.0 * p00) / (2.0 * h * h);
    a[4] = (ppp - pp0 - p0p + p00) / (h * h);
}

// Deviation of the equilibrium populations for the wall state (drho, dE) and
// wall velocity (ux, uy), from the double collision constants kd.
inline void wall_equilibrium(const Coef<double> &kd, double drho, double dE, double ux, double uy, double f[Q])
{
    const double rho = 1.0 + drho;
    equilibrium_dev(drho, dE, rho * ux, rho * uy, kd, f);
}

// The four sides' wall arguments (west, east, south, north): kinds, wall
// velocity and temperature terms, zero-flux constants and the correction
// polynomial of each entering link.  D: lbm13_derive's constants; kd: the
// double collision constants of the same lattice.
template <typename C>
void wall_coef(const lbm13_params &p, const double *D, const lbm13_boundary &b, const Coef<double> &kd,
               WallArgs<C> *w)
{
    const lbm13_wall *src[4] = {&b.west, &b.east, &b.south, &b.north};
    for (int s = 0; s < 4; ++s) {
        const lbm13_wall &in = *src[s];
        WallArgs<C> &o = w[s];
        const double ux = s <= EAST ? 0.0 : in.u_t, uy = s <= EAST ? in.u_t : 0.0;
        o.kind = in.kind;
        o.needs_data = in.kind == WALL_MIXED || (in.kind == WALL_BB && in.u_t != 0.0);
        o.ux = C(ux);
        o.uy = C(uy);
        o.base = C(26.0 * in.T - 28.0);
        o.eT = C(26.0 * (in.T - (p.E0 + 28.0) / 26.0));
        o.mass_flux = in.kind == WALL_MIXED && b.wall_density == LBM13_WALL_DENSITY_ZERO_FLUX;
        o.ke = C(13.0 * in.u_t * in.u_t);
        // zero-flux density: even parts of the unit-density wall equilibrium on
        // the outgoing unit and distance-2 normal links
        double e[Q];
        wall_equilibrium(kd, 0.0, 26.0 * (in.T - (p.E0 + 28.0) / 26.0) + 13.0 * (ux * ux + uy * uy), ux, uy, e);
        const int ja = s == WEST ? 3 : s == EAST ? 1 : s == SOUTH ? 4 : 2;
        const int jb = s == WEST ? 11 : s == EAST ? 9 : s == SOUTH ? 12 : 10;
        const double zf_e = 0.5 * (e[ja] + e[copp(ja)]) + (e[jb] + e[copp(jb)]);
        const double zf_den = D[22 + 1] + 2.0 * D[22 + 9] + zf_e;
        o.zf_e = C(zf_e);
        o.zf_den = C(zf_den);
        o.zf_inv = C(1.0 / zf_den);
        o.lin = o.quad = 0;
        for (int i = 0; i < 4; ++i) {
            const int j = wall_link(s, i), jn = copp(j);
            const bool normal = s <= EAST ? cvy(j) == 0 : cvx(j) == 0;
            const bool abb = in.kind == WALL_MIXED && normal;
            double a[5];
            quadratic_coefficients(
                [&](double dr, double de) {
                    double f[Q];
                    wall_equilibrium(kd, dr, de, ux, uy, f);
                    return abb ? f[j] + f[jn] : f[j] - f[jn];
                },
                a);
            if (in.u_t == 0.0) a[3] = a[4] = 0.0;  // linear in rho and E without momentum
            for (int m = 0; m < 5; ++m) o.poly[i][m] = C(a[m]);
            o.lin |= (a[0] != 0.0 || a[1] != 0.0 || a[2] != 0.0 ? 1 : 0) << i;
            o.quad |= (a[3] != 0.0 || a[4] != 0.0 ? 1 : 0) << i;
        }
        if (!o.needs_data) o.lin = o.quad = 0;
    }
    // a corner diagonal crosses both walls and takes both walls' corrections
    // for its link (their slots above), each at its own wall's state
}

} // namespace lbm13

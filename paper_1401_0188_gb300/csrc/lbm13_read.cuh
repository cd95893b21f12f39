// lbm13_read.cuh -- what the read-outs and reductions take from one node, shared
// by lbm13_aux.cu and lbm13_noalloc.cu (the same code, so the same values).
#pragma once

#include "lbm13_internal.h"

namespace lbm13 {

template <typename T>
__device__ __forceinline__ void load_node(const ReadArgs<T> &a, long long idx, T (&f)[Q])
{
#pragma unroll
    for (int j = 0; j < Q; ++j) f[j] = a.f[(long long)j * a.plane + idx];
}
template <typename T>
__device__ __forceinline__ void widen(const T (&f)[Q], double (&g)[Q])
{
#pragma unroll
    for (int j = 0; j < Q; ++j) g[j] = double(f[j]);
}

// What the reductions take from one node: deviations of rho, E and the momentum,
// velocity, deviations of T and p (read half-way), and its non-finite populations.
struct NodeDev {
    double rho, E, jx, jy, ux, uy, T, p, bad;
};

// In FP64: the read-out of FP64 lattices, and of nodes that the integer one does not
// take.  Populations are summed as they are, so that a small velocity beside large
// deviations of density or temperature keeps its digits (integers of the node's
// largest population lost up to 8,000 times what FP64 loses there).  The quotients by
// rho near 1 share one reciprocal and take a residual correction each, within an ulp's
// 2^-50 of the division.  2048^2 FP64, all 13 moments; rho, u and T; one residual: 843, 640
// and 1411 us with four divisions a node, 283, 147 and 438 in integers, 459, 459 and
// 785 so (7 us an FP64 operation a node).
//
// u_x, u_y and the deviations of T and p, read half-way through the force and the
// source, from those of rho, E and the momentum; over(x) = x / rho.
template <typename T, typename Over>
LBM13_HD void macro_quotients(const ReadArgs<T> &a, double drho, double dE, double jx, double jy, Over over, double &ux,
                              double &uy, double &dT, double &dp)
{
    double k2;  // |j|^2 / rho
    if (a.force) {
        const double h = 0.5 * (1.0 + drho - a.rho_ref);
        ux = over(jx - h * a.gx);
        uy = over(jy - h * a.gy);
        k2 = over(fma(jx, jx, jy * jy));
    } else {
        ux = over(jx);
        uy = over(jy);
        k2 = fma(jx, ux, jy * uy);
    }
    const double s = fma(28.0, drho, dE), q = s * (1.0 / 26.0);
    dp = fma(-0.5, k2, fma(fma(-26.0, q, s), 1.0 / 26.0, q)) - 0.5 * a.heat;
    dT = over(fma(-a.rest.T0, drho, dp));
}
template <typename T>
__host__ __device__ __noinline__ void macro_far(const ReadArgs<T> &a, double drho, double dE, double jx, double jy,
                                                double &ux, double &uy, double &dT, double &dp)
{
    const double rho = 1.0 + drho;
    macro_quotients(a, drho, dE, jx, jy, [&](double x) { return x / rho; }, ux, uy, dT, dp);
}
template <typename T>
LBM13_HD void macro_dev(const ReadArgs<T> &a, double drho, double dE, double jx, double jy, double &ux, double &uy,
                        double &dT, double &dp)
{
    const double rho = 1.0 + drho;
    if (uint32_t(fx_bits(rho) >> 32) - 0x3fe00000u >= 0x200000u) {  // not in [0.5, 2)
        double v[4];
        macro_far(a, drho, dE, jx, jy, v[0], v[1], v[2], v[3]);
        ux = v[0];
        uy = v[1];
        dT = v[2];
        dp = v[3];
        return;
    }
    const double inv = recip(rho);
    macro_quotients(a, drho, dE, jx, jy,
                    [&](double x) {
                        const double q = x * inv;
                        return fma(fma(-q, rho, x), inv, q);
                    },
                    ux, uy, dT, dp);
}

template <typename T>
__device__ __forceinline__ NodeDev node_dev_wide(const ReadArgs<T> &a, const double (&f)[Q])
{
    NodeDev o;
    o.bad = 0.0;
    uint32_t M = fx_mag(f[0]);
#pragma unroll
    for (int j = 1; j < Q; ++j) M = M > fx_mag(f[j]) ? M : fx_mag(f[j]);
    if (M >= 0x7ff00000u) {
#pragma unroll
        for (int j = 0; j < Q; ++j) o.bad += isfinite(f[j]) ? 0.0 : 1.0;
    }
    Mom<double> d;
    forward(f, d);
    o.rho = d.rho;
    o.E = d.E;
    o.jx = d.jx;
    o.jy = d.jy;
    macro_dev(a, d.rho, d.E, d.jx, d.jy, o.ux, o.uy, o.T, o.p);
    return o;
}
template <typename T>
__device__ __noinline__ NodeDev node_dev_plain(const ReadArgs<T> &a, const T (&raw)[Q])
{
    double f[Q];
    widen(raw, f);
    return node_dev_wide(a, f);
}

__device__ __forceinline__ NodeDev node_dev(const ReadArgs<double> &a, long long idx)
{
    double f[Q];
    load_node(a, idx, f);
    return node_dev_wide(a, f);
}
__device__ __forceinline__ NodeDev node_dev(const ReadArgs<float> &a, long long idx)
{
    float f[Q];
    load_node(a, idx, f);
    FxSums s;
    FxMacro m;
    if (!fx_sums(f, s) || !fx_macro(s, a.fx, m)) {
        float g[Q];  // f itself stays in registers
#pragma unroll
        for (int j = 0; j < Q; ++j) g[j] = f[j];
        return node_dev_plain(a, g);
    }
    NodeDev o;
    o.rho = s.value(m.drho);
    o.E = s.energy();
    o.jx = s.value(s.jx());
    o.jy = s.value(s.jy());
    o.ux = s.value(m.u);
    o.uy = s.value(m.v);
    o.T = s.value(m.T);
    o.p = s.value(m.p);
    o.bad = 0.0;
    return o;
}

} // namespace lbm13

#pragma once
// The operator of the velocity-Exner form at one entry of a stacked vector
// [u; v; pi] (exner.cu: the equations).
#include "krylov_impl.cuh"

namespace wrc {

namespace {

// M q at the active points: the frozen-coefficient operator (advection by
// the state's velocity, pressure gradient, pi times the divergence,
// Coriolis, friction, viscosity) plus, for the exact Jacobian, the terms of
// the state's gradients.
// Entry e of M q (e = f n + i: field f at active point i; M the exact
// Jacobian with full, else the frozen-coefficient operator): the own field's
// collocation derivatives at the point's stencil levels and the cross terms
// of the other fields (the lattices a.Lq hold q with its ghost values; mw:
// the point's packed index and stencil levels).
template <int P>
__device__ __forceinline__ double ex_entry(const ExArgs& a, uint32_t mw, int f, int i) {
    const long long ld = a.ld;
    const double* d = a.d;
    const double u = a.f[0][i], v = a.f[1][i];
    const int p = meta_pos(mw);
    const double du = a.Lq[0][p], dv = a.Lq[1][p];
    if (f == 0) {
        double dx, dy, lap;
        point_derivs<double, P>(a.Lq[0], mw, a.g, a.c1J, a.c2J, dx, dy, lap);
        const double dpx = point_d1<double, P>(a.Lq[2], mw, a.g, a.c1J, 0);
        double J = -(u * dx + v * dy) - a.C * dpx + a.fc * dv - a.r * du + a.nu * lap;
        if (a.full) J -= du * d[i] + dv * d[ld + i];
        return J;
    }
    if (f == 1) {
        double dx, dy, lap;
        point_derivs<double, P>(a.Lq[1], mw, a.g, a.c1J, a.c2J, dx, dy, lap);
        const double dpy = point_d1<double, P>(a.Lq[2], mw, a.g, a.c1J, 1);
        double J = -(u * dx + v * dy) - a.C * dpy - a.fc * du - a.r * dv + a.nu * lap;
        if (a.full) J -= du * d[2 * ld + i] + dv * d[3 * ld + i];
        return J;
    }
    const double dpx = point_d1<double, P>(a.Lq[2], mw, a.g, a.c1J, 0);
    const double dpy = point_d1<double, P>(a.Lq[2], mw, a.g, a.c1J, 1);
    const double dux = point_d1<double, P>(a.Lq[0], mw, a.g, a.c1J, 0);
    const double dvy = point_d1<double, P>(a.Lq[1], mw, a.g, a.c1J, 1);
    double J = -(u * dpx + v * dpy) - a.f[2][i] * (dux + dvy);
    if (a.full) J -= (du * d[4 * ld + i] + dv * d[5 * ld + i]) + a.Lq[2][p] * (d[i] + d[3 * ld + i]);
    return J;
}

// Field and point of a stacked entry.
__device__ __forceinline__ void ex_split(long long e, int n, int& f, int& i) {
    f = e >= 2LL * n ? 2 : (e >= n ? 1 : 0);
    i = (int)(e - (long long)f * n);
}

// Absolute sum of the operator's row at entry (f, i): |M q| <= it times max |q|.
template <int P>
__device__ __forceinline__ double ex_row_bound(const ExArgs& a, uint32_t mw, int f, int i) {
    double d1 = 0.0, d2 = -dd_d2(P, 0);
#pragma unroll
    for (int o = 1; o <= dd_reach1(P); ++o) d1 += 2.0 * (dd_d1(P, o) < 0 ? -dd_d1(P, o) : dd_d1(P, o));
#pragma unroll
    for (int o = 1; o <= P; ++o) d2 += 2.0 * (dd_d2(P, o) < 0 ? -dd_d2(P, o) : dd_d2(P, o));
    const int shx = a.g.J - meta_jx(mw), shy = a.g.J - meta_jy(mw);
    const double dx = d1 * pow2_down(a.c1J, shx), dy = d1 * pow2_down(a.c1J, shy);
    const long long ld = a.ld;
    const double* d = a.d;
    double s = fabs(a.f[0][i]) * dx + fabs(a.f[1][i]) * dy;
    if (f == 2) {
        s += fabs(a.f[2][i]) * (dx + dy);
        if (a.full) s += fabs(d[4 * ld + i]) + fabs(d[5 * ld + i]) + fabs(d[i] + d[3 * ld + i]);
    } else {
        s += fabs(a.C) * (f == 0 ? dx : dy) + fabs(a.fc) + fabs(a.r) +
             a.nu * d2 * (pow2_down(a.c2J, 2 * shx) + pow2_down(a.c2J, 2 * shy));
        if (a.full) s += fabs(d[2 * f * ld + i]) + fabs(d[(2 * f + 1) * ld + i]);
    }
    return s;
}

}  // namespace

}  // namespace wrc

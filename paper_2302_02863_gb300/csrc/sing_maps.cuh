// The singular rules of Sec. 4 in 2D: region maps, and what of a 4D point does not
// depend on the element pair (singular.cu, grad.cu).
#pragma once

#include <cmath>

#include "vfd_internal.h"

namespace vfd {

// region maps divided by xi: xhat = xi a, yhat = xi b (vertex: T_V^(1,2)
// eq. e:map-v; edge: T_E^(1..5) Sec. 4.2), with the eta-Jacobian factor
__device__ __forceinline__ void map_ve(int type, int reg, double e1, double e2, double e3, double *a, double *b,
                                       double &jac)
{
    if (type == 1) {
        if (reg == 0) { a[0] = 1.0; a[1] = e1; b[0] = e2; b[1] = e2 * e3; }
        else { a[0] = e2; a[1] = e2 * e3; b[0] = 1.0; b[1] = e1; }
        jac = e2;
        return;
    }
    switch (reg) {
    case 0: a[0] = 1.0; a[1] = e1 * e3; b[0] = 1.0 - e1 * e2; b[1] = e1 * (1.0 - e2); jac = e1 * e1; break;
    case 1: a[0] = 1.0; a[1] = e1; b[0] = 1.0 - e1 * e2 * e3; b[1] = e1 * e2 * (1.0 - e3); jac = e1 * e1 * e2; break;
    case 2: a[0] = 1.0 - e1 * e2; a[1] = e1 * (1.0 - e2); b[0] = 1.0; b[1] = e1 * e2 * e3; jac = e1 * e1 * e2; break;
    case 3: a[0] = 1.0 - e1 * e2 * e3; a[1] = e1 * e2 * (1.0 - e3); b[0] = 1.0; b[1] = e1; jac = e1 * e1 * e2; break;
    default: a[0] = 1.0 - e1 * e2 * e3; a[1] = e1 * (1.0 - e2 * e3); b[0] = 1.0; b[1] = e1 * e2; jac = e1 * e1 * e2; break;
    }
}

// identical maps T_I^(1..3) (Sec. 4.3; region 2 with the factor eta1 on
// xhat_2, region 3 scaled difference (-eta3, 1-eta3)); dr = (xhat - yhat)/(xi eta1 eta2)
__device__ __forceinline__ void map_id(int reg, double e1, double e2, double e3, double *a, double *b, double *dr)
{
    if (reg == 0) {
        a[0] = 1.0; a[1] = 1.0 - e1 + e1 * e2; b[0] = 1.0 - e1 * e2 * e3; b[1] = 1.0 - e1;
        dr[0] = e3; dr[1] = 1.0;
    } else if (reg == 1) {
        a[0] = 1.0; a[1] = e1 * (1.0 - e2 + e2 * e3); b[0] = 1.0 - e1 * e2; b[1] = e1 * (1.0 - e2);
        dr[0] = 1.0; dr[1] = e3;
    } else {
        a[0] = 1.0 - e1 * e2 * e3; a[1] = e1 * (1.0 - e2 * e3); b[0] = 1.0; b[1] = e1 * (1.0 - e2);
        dr[0] = -e3; dr[1] = 1.0 - e3;
    }
}

// vertex pairs have 2 regions, edge pairs 5, identical pairs 3 (ns^4 points each);
// tables hold the types one after another
__device__ __forceinline__ int sing_regions(int type) { return type == 1 ? 2 : (type == 2 ? 5 : 3); }
// first table entry of a type, in units of ns^4
__device__ __forceinline__ int sing_first(int type) { return type == 1 ? 0 : (type == 2 ? 2 : 7); }

// a 4D point (zeta, eta1, eta2 or t, eta3) of region reg
struct SingPoint {
    double xi;    // zeta^(1/c): the mapped points are xi a and xi b
    double w;     // map Jacobian and the constants of the rule, without Gauss weights and cell Jacobians
    double f[5];  // basis differences over xi (f[0] is minus the sum of the others, not set)
    // (2 sbar - S) q + (2 - S) l in base 2 = cst - (b_x + b_y) nu / ln 2, with S = 2 (b_x + b_y) - 2,
    // q = ln zeta / c (+ ln t / c2) and l = ln eta1 for identical pairs
    double nu, cst;
};

// a, b: mapped points over xi; d: coefficients of the scaled difference x - y
// (J_P (d0, d1) - J_Q (d2, d3))
__device__ __forceinline__ SingPoint sing_point(int type, int reg, double sbar, double zeta, double e1, double e2,
                                                double e3, double *a, double *b, double *d)
{
    SingPoint p;
    const double c = 4.0 - 2.0 * sbar, c2 = 2.0 - 2.0 * sbar, lz = log(zeta);
    double q = lz / c, l = 0.0;
    p.xi = exp(q);
    for (int i = 0; i < 5; ++i) p.f[i] = 0.0;
    if (type == 3) {
        const double lt = log(e2);
        double dr[2];
        map_id(reg, e1, exp(lt / c2), e3, a, b, dr);
        d[0] = dr[0];
        d[1] = dr[1];
        d[2] = d[3] = 0.0;
        p.w = 2.0 / (c * c2);   // the mirror regions T_I^(4..6) double the sum
        q += lt / c2;
        l = log(e1);
        p.f[1] = dr[0] - dr[1];
        p.f[2] = dr[1];
    } else {
        double jac;
        map_ve(type, reg, e1, e2, e3, a, b, jac);
        for (int i = 0; i < 2; ++i) {
            d[i] = a[i];
            d[2 + i] = b[i];
        }
        p.w = jac / c;
        p.f[1] = type == 1 ? a[0] - a[1] : (a[0] - a[1]) - (b[0] - b[1]);
        p.f[2] = a[1];
        p.f[3] = type == 1 ? -(b[0] - b[1]) : -b[1];
        p.f[4] = type == 1 ? -b[1] : 0.0;
    }
    p.nu = -2.0 * (q + l);
    p.cst = ((2.0 * sbar + 2.0) * q + 4.0 * l) * 1.4426950408889634;
    return p;
}

// v 2^n as an integer, in the bits of an FP64 table entry
__device__ __forceinline__ double fx_bits(double v, int n) { return __longlong_as_double(__double2ll_rn(ldexp(v, n))); }

// nu and cst grow with the number of Gauss points and as s_bar nears 1: whether they
// fit the fixed-point exponent
inline bool sing_fixed_fits(const MeshData &m, double s_bar)
{
    const double lg = std::fabs(std::log(m.gl_min)), c = 4.0 - 2.0 * s_bar, c2 = 2.0 - 2.0 * s_bar;
    const double q = lg * (1.0 / c + 1.0 / c2);
    return c2 > 0.0 && 2.0 * (q + lg) < 60.0 && 1.45 * (std::fabs(2.0 * s_bar + 2.0) * q + 4.0 * lg) < 200.0;
}

}  // namespace vfd

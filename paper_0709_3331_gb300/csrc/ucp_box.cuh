// ucp_box.cuh -- a box's geometry from its key prefix, its moments from its sums.
#pragma once

#include "ucp_internal.cuh"

namespace ucp {

__device__ __forceinline__ unsigned int compact3(unsigned long long x)
{
    x &= 0x1249249249249249ull;
    x = (x | (x >> 2)) & 0x10c30c30c30c30c3ull;
    x = (x | (x >> 4)) & 0x100f00f00f00f00full;
    x = (x | (x >> 8)) & 0x001f0000ff0000ffull;
    x = (x | (x >> 16)) & 0x001f00000000ffffull;
    x = (x | (x >> 32)) & 0x1fffffull;
    return (unsigned int)x;
}

// cube of the cloud that owns the box starting at sorted position i
__device__ __forceinline__ Cube cube_of(const Cube* __restrict__ cubes, const Tree& t, int i)
{
    return cubes[t.cloud ? t.cloud[i] : 0];
}

// geometric box centre: lo + (cell + 1/2) * side, side = L 2^-depth
__device__ __forceinline__ void box_centre(const Cube& cb, unsigned long long cell, int d,
                                           double ctr[3], double* side)
{
    double s = ldexp(cb.L, -d);
    *side = s;
    unsigned int ic[3] = {compact3(cell), compact3(cell >> 1), compact3(cell >> 2)};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        double lo = __dsub_rn(cb.c[a], __dmul_rn(cb.L, 0.5));
        ctr[a] = __dadd_rn(lo, __dmul_rn(__dadd_rn((double)ic[a], 0.5), s));
    }
}

// The same with what rounding took from z: the exact centre is z + rho (to 2^-106 L; for
// the cube's corner as it is stored).
__device__ __forceinline__ void box_centre_exact(const Cube& cb, unsigned long long cell, int d,
                                                 double z[3], double rho[3])
{
    const double s = ldexp(cb.L, -d);
    const unsigned int ic[3] = {compact3(cell), compact3(cell >> 1), compact3(cell >> 2)};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const double lo = __dsub_rn(cb.c[a], __dmul_rn(cb.L, 0.5));
        const double k = __dadd_rn((double)ic[a], 0.5), t = __dmul_rn(k, s);
        z[a] = __dadd_rn(lo, t);
        // Dekker's fast two-sum: the larger first (by exponents, on the integer units)
        const bool lo_first = (__double2hiint(lo) & 0x7fffffff) >= (__double2hiint(t) & 0x7fffffff);
        const double p = lo_first ? lo : t, q = lo_first ? t : lo;
        rho[a] = __dadd_rn(__dsub_rn(q, __dsub_rn(z[a], p)), __fma_rn(k, s, -t));
    }
}

// FP64 moments of one box from sums about its exact geometric centre z + rho:
//   a = {S0, M, sum|q|y (3), sum q y (3), sum q y y^T (6)},  y = x - z - rho.
// The expansion centre is the |q|-weighted centroid c = z + rho + e, e = sum|q|y / S0
// (0 when S0 = 0); shifting to c: D = sum q y - M e,
// Q = sum q y y^T - (sum q y) e^T - e (sum q y)^T + M e e^T.  delta = |c - z|.
__device__ __forceinline__ void finish_box(const double* a, const double z[3], const double rho[3],
                                           double* __restrict__ m, double* __restrict__ delta)
{
    double S0 = a[0], M = a[1];
    double e[3];
    const double inv = S0 > 0.0 ? 1.0 / S0 : 0.0;
    for (int k = 0; k < 3; ++k) e[k] = a[2 + k] * inv;
    double d[3];
    for (int k = 0; k < 3; ++k) d[k] = a[5 + k];
    for (int k = 0; k < 3; ++k) m[MC + k] = z[k] + (e[k] + rho[k]);
    m[MM] = M;
    for (int k = 0; k < 3; ++k) m[MD + k] = d[k] - M * e[k];
    const int ia[6] = {0, 0, 0, 1, 1, 2}, ib[6] = {0, 1, 2, 1, 2, 2};
    for (int k = 0; k < 6; ++k)
        m[MQ + k] = a[8 + k] - d[ia[k]] * e[ib[k]] - e[ia[k]] * d[ib[k]] + M * e[ia[k]] * e[ib[k]];
    m[MS0] = S0;
    // delta = |c - z| rounded like the definition: c is stored first, then differenced
    double ex = __dsub_rn(m[MC + 0], z[0]);
    double ey = __dsub_rn(m[MC + 1], z[1]);
    double ez = __dsub_rn(m[MC + 2], z[2]);
    *delta = __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(ex, ex), __dmul_rn(ey, ey)),
                                  __dmul_rn(ez, ez)));
    m[MT] = -0.5 * (m[MQ] + m[MQ + 3] + m[MQ + 5]);
}

}  // namespace ucp

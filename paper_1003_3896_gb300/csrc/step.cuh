// step.cuh -- arithmetic of a substep that more than one kernel performs: the
// external field, a cluster's moments and frame, kick and drift.  Roundings are
// spelt out (no multiply-add left to the compiler's choice), so the kernels give
// the same bits.
#pragma once

#include "nb_internal.cuh"
#include "split.cuh"

namespace nb {

// Acceleration of the smooth field of eq. 3, a = -grad Phi, for the
// Miyamoto-Nagai disk plus Plummer bulge potential
//   Phi = -G Md / sqrt(R^2 + (ad + sqrt(z^2 + bd^2))^2) - G Mb / sqrt(r^2 + ab^2).
// Added to ax, ay, az.  Written with three reciprocal square roots and no
// division: the FP64 pipe of this part runs at a small fraction of the FP32
// rate, and a double division or square root costs several times an rsqrt.
__device__ __forceinline__ void field_accel(const ExtField &e, double x, double y, double z,
                                            double &ax, double &ay, double &az)
{
    // the inverse square-root powers refined in double from float estimates
    // (split.cuh: the FP64 pipe carries the kick here)
    const double R2 = __fma_rn(x, x, __dmul_rn(y, y)), r2 = __fma_rn(z, z, R2);
    const double s2 = __fma_rn(z, z, __dmul_rn(e.bd, e.bd));
    const double rs = rsqrt_pow<true>(s2);         // 1 / sqrt(z^2 + bd^2)
    const double q = __fma_rn(s2, rs, e.ad);       // ad + sqrt(z^2 + bd^2)
    const double kd = __dmul_rn(__dmul_rn(e.G, e.Md), rsqrt_pow<false>(__fma_rn(q, q, R2)));
    const double kb =
        __dmul_rn(__dmul_rn(e.G, e.Mb), rsqrt_pow<false>(__fma_rn(e.ab, e.ab, r2)));
    double kh = 0.0;   // softened central point mass
    if (e.Mbh > 0)
        kh = __dmul_rn(__dmul_rn(e.G, e.Mbh), rsqrt_pow<false>(__dadd_rn(r2, e.eps2bh)));
    const double kr = __dadd_rn(kb, kh), kx = __dadd_rn(kd, kr);
    ax = __fma_rn(-kx, x, ax);
    ay = __fma_rn(-kx, y, ay);
    az = __fma_rn(-__fma_rn(__dmul_rn(kd, q), rs, kr), z, az);
}

// A body's part of its cluster's moments.
__device__ __forceinline__ void moment_add(double (&v)[5], double m, double x, double y, double z)
{
    v[0] = __dadd_rn(v[0], m);
    v[1] = __fma_rn(m, x, v[1]);
    v[2] = __fma_rn(m, y, v[2]);
    v[3] = __fma_rn(m, z, v[3]);
    v[4] = __fma_rn(m, __fma_rn(z, z, __fma_rn(y, y, __dmul_rn(x, x))), v[4]);
}

// Velocity after a kick, position after a drift, one component.
__device__ __forceinline__ double moved(double h, double rate, double v)
{
    return __fma_rn(h, rate, v);
}

// Frame of a cluster from its moments (sum m, m x, m y, m z, m r^2): the
// mass-weighted centre and mean square radius.  No near-pair radius yet (set by
// frame_scale_kernel when the plan runs the near-pair pass).
__device__ __forceinline__ Frame frame_of(const double (&v)[5], double eps2)
{
    Frame f;
    const double M = v[0];
    const double iM = M > 0 ? 1.0 / M : 0.0;   // one division, four products
    f.cx = __dmul_rn(v[1], iM);
    f.cy = __dmul_rn(v[2], iM);
    f.cz = __dmul_rn(v[3], iM);
    const double c2 = __fma_rn(f.cz, f.cz, __fma_rn(f.cy, f.cy, __dmul_rn(f.cx, f.cx)));
    const double r2 = M > 0 ? __fma_rn(v[4], iM, -c2) : 0.0;
    f.r2rms = r2 > 0 ? r2 : 0.0;
    f.th2 = (float)eps2;
    f.dth = 0.f;
    f.hx = INFINITY;
    return f;
}

}  // namespace nb

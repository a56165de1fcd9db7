// esmm_vjp.cuh -- reverse sweeps shared by the RHD and RMHD adjoints: the
// logarithmic mean and the WENO edge values.
#pragma once

#include "esmm_device.cuh"

namespace esmm {

// Adjoint of logmean's mean (gm), added to the adjoints of the values and logs.
__device__ __forceinline__ void logmean_vjp(double a, double b, double la, double lb, double thr, double gm, double &ga,
                                            double &gb, double &gla, double &glb)
{
    const double d = b - a, s = b + a;
    if (d * d < thr * s * s) {
        // mean = s/(2F(u)), u = r^2, r = d/s: d mean = ds/(2F) - (F'/F^2) r (dd - r ds)
        const double is = __drcp_rn(s), r = d * is, u = r * r;
        const double F = 1.0 + u * (1.0 / 3.0 + u * (1.0 / 5.0 + u * (1.0 / 7.0)));
        const double F1 = 1.0 / 3.0 + u * (2.0 / 5.0 + u * (3.0 / 7.0));
        const double iF = __drcp_rn(F);
        const double c0 = 0.5 * iF * gm, c1 = F1 * iF * iF * r * gm;
        ga += c0 + c1 * (1.0 + r);
        gb += c0 - c1 * (1.0 - r);
    } else {
        const double idl = __drcp_rn(lb - la), g = gm * idl, m = d * idl * g;
        ga -= g;
        gb += g;
        gla += m;
        glb -= m;
    }
}

// Adjoint of one WENO edge value from its stencil V (upwind first), g the value's
// adjoint: with r_k = 1/(eps + b_k) and w_k = d_k r_k^2 / sum,
// dv = sum_k w_k dq_k - 2 w_k (q_k - v) r_k db_k.
__device__ __forceinline__ void weno5_vjp(double V0, double V1, double V2, double V3, double V4, double eps, double g,
                                          double gV[5])
{
    const double c = 13.0 / 12.0;
    const double t0 = V0 - 2.0 * V1 + V2, t1 = V1 - 2.0 * V2 + V3, t2 = V2 - 2.0 * V3 + V4;
    const double r0 = V0 - 4.0 * V1 + 3.0 * V2, r1 = V1 - V3, r2 = 3.0 * V2 - 4.0 * V3 + V4;
    const double e0 = eps + c * t0 * t0 + 0.25 * r0 * r0, e1 = eps + c * t1 * t1 + 0.25 * r1 * r1,
                 e2 = eps + c * t2 * t2 + 0.25 * r2 * r2;
    const double i0 = __drcp_rn(e0), i1 = __drcp_rn(e1), i2 = __drcp_rn(e2);
    const double a0 = 0.1 * i0 * i0, a1 = 0.6 * i1 * i1, a2 = 0.3 * i2 * i2, ia = __drcp_rn(a0 + a1 + a2);
    const double q0 = (2.0 * V0 - 7.0 * V1 + 11.0 * V2) * (1.0 / 6.0), q1 = (-V1 + 5.0 * V2 + 2.0 * V3) * (1.0 / 6.0),
                 q2 = (2.0 * V2 + 5.0 * V3 - V4) * (1.0 / 6.0);
    const double w0 = a0 * ia * g, w1 = a1 * ia * g, w2 = a2 * ia * g, v = (a0 * q0 + a1 * q1 + a2 * q2) * ia;
    const double h0 = -2.0 * w0 * (q0 - v) * i0, h1 = -2.0 * w1 * (q1 - v) * i1, h2 = -2.0 * w2 * (q2 - v) * i2;
    const double T0 = 2.0 * c * t0 * h0, T1 = 2.0 * c * t1 * h1, T2 = 2.0 * c * t2 * h2;
    const double R0 = 0.5 * r0 * h0, R1 = 0.5 * r1 * h1, R2 = 0.5 * r2 * h2;
    gV[0] = w0 * (1.0 / 3.0) + T0 + R0;
    gV[1] = -w0 * (7.0 / 6.0) - w1 * (1.0 / 6.0) - 2.0 * T0 - 4.0 * R0 + T1 + R1;
    gV[2] = w0 * (11.0 / 6.0) + w1 * (5.0 / 6.0) + w2 * (1.0 / 3.0) + T0 + 3.0 * R0 - 2.0 * T1 + T2 + 3.0 * R2;
    gV[3] = w1 * (1.0 / 3.0) + w2 * (5.0 / 6.0) + T1 - R1 - 2.0 * T2 - 4.0 * R2;
    gV[4] = -w2 * (1.0 / 6.0) + T2 + R2;
}
__device__ __forceinline__ void weno3_vjp(double V0, double V1, double V2, double eps, double g, double gV[3])
{
    const double d0 = V1 - V0, d1 = V2 - V1;
    const double i0 = __drcp_rn(eps + d0 * d0), i1 = __drcp_rn(eps + d1 * d1);
    const double a0 = (1.0 / 3.0) * i0 * i0, a1 = (2.0 / 3.0) * i1 * i1, ia = __drcp_rn(a0 + a1);
    const double q0 = (-V0 + 3.0 * V1) * 0.5, q1 = (V1 + V2) * 0.5, v = (a0 * q0 + a1 * q1) * ia;
    const double w0 = a0 * ia * g, w1 = a1 * ia * g;
    const double h0 = -4.0 * w0 * (q0 - v) * i0 * d0, h1 = -4.0 * w1 * (q1 - v) * i1 * d1;
    gV[0] = -0.5 * w0 - h0;
    gV[1] = 1.5 * w0 + 0.5 * w1 + h0 - h1;
    gV[2] = 0.5 * w1 + h1;
}
// adjoint of the jump (right minus left edge value) of one field from its WW + 1
// stencil values
template <int WW>
__device__ __forceinline__ void weno_jump_vjp(const double *V, double eps, double g, double *gV)
{
    double a[WW], b[WW];
    if constexpr (WW == 5) {
        weno5_vjp(V[0], V[1], V[2], V[3], V[4], eps, -g, a);
        weno5_vjp(V[5], V[4], V[3], V[2], V[1], eps, g, b);
    } else {
        weno3_vjp(V[0], V[1], V[2], eps, -g, a);
        weno3_vjp(V[3], V[2], V[1], eps, g, b);
    }
#pragma unroll
    for (int k = 0; k <= WW; ++k) gV[k] = (k < WW ? a[k < WW ? k : 0] : 0.0) + (k > 0 ? b[k > 0 ? WW - k : 0] : 0.0);
}

}  // namespace esmm

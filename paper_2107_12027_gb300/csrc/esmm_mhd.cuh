// esmm_mhd.cuh -- device arithmetic and kernels of the RMHD scheme (Duan &
// Tang, arXiv 2107.12027): primitive recovery, the two-point EC flux with its
// Godunov-Powell term, the scaled eigenvectors of the symmetrized system, the
// ES interface flux, the Powell source in the update, and the CFL radius.
//
// State: cons [8][N] = J (D, m_1, m_2, m_3, E, B_1, B_2, B_3), primitives
// (rho, v_1, v_2, v_3, p, B_1, B_2, B_3).  Node data extend the RHD layout of
// esmm_device.cuh (indices 0..13 keep their meaning) by u_3 and B_1..B_3, so
// the mesh, temporal-metric and totals kernels serve both systems.
// Device arithmetic and the templated kernels; the 2D instantiations live in
// esmm_mhd.cu and the 3D kernels (esmm_3d.cu) reuse the arithmetic.
#pragma once

#include <type_traits>

#include "esmm_device.cuh"
#include "esmm_launch.h"

namespace esmm {

enum { QM_UZ = NQ, QM_B1, QM_B2, QM_B3, NQM };   // 18 node arrays (NQ_MHD)
// FP32 copies for the mixed form's flux kernel, written by the FP64 node pass (an
// interface reads 26 nodes' values: converting them there took about as many instructions
// as its arithmetic); RLO, BLO: the FP64 rests of rho and beta
enum { QM32_R = 0, QM32_B, QM32_LNR, QM32_LNB, QM32_W, QM32_U0, QM32_U1, QM32_U2, QM32_B0, QM32_B1, QM32_B2, QM32_RLO,
       QM32_BLO, NQM32 };
static_assert(NQM32 == NQ32_MHD, "the allocation of the FP32 copies");
constexpr int NFM = 10;                          // interface values per direction: F[8], J xi_t, B~ (NF_MHD)

// ---------------------------------------------------------------------------
// Primitive recovery (FP64).  The root in Z = rho h W^2 of, with S = m.B,
//   v.B = S/Z,  |v|^2 = (|m|^2 + (2Z + |B|^2) S^2/Z^2)/(Z + |B|^2)^2,
//   p = (Gamma-1)/Gamma (Z/W^2 - D/W),
//   f(Z) = Z - p + |B|^2 (1 + |v|^2)/2 - S^2/(2 Z^2) - E,
// a trial Z with |v|^2 >= 1 lying below the root.  As in cons2prim_gg: an FP32 Newton
// iteration gives Z to about 1e-7, one FP64 step of third order lands on the root to
// rounding (the last where it is below 3e-6 of Z (1 - v^2), the length on which f bends, and
// its second-order part below 3e-6 of it), and where that fails three times c2p_loop_mhd, FP64 Newton with
// bisection on [0, Gamma E], which stops when a step moves Z by at most 1e-15 (E + Z), or
// where |f| <= 2e-15 (E + Z), f's rounding level (a root, whose tiny steps the open
// bracket would otherwise reject).  The FP32 parts work in units of E (converted over powers of
// two, so that E^2 and E^3 stay in FP32's range).
// Z0: warm start (ignored outside the bracket).  Measured: the node pass of 512^2 nodes 214 ->
// 146 us, mixed rotor steps 3.71 -> 3.05 ms (with the speeds' pass in 80 registers).
// Returns 0, 1 (non-admissible) or 2 (iteration cap).
__device__ __forceinline__ float c2p_estimate_mhd(float g, float gam, float D, float m2, float B2, float S2, float z0)
{
    float lo = 0.0f, hi = gam, Z = z0;
#pragma unroll 1
    for (int it = 0; it < 24; ++it) {
        const float iZ = __frcp_rn(Z), q = __frcp_rn(Z + B2), t = S2 * iZ * iZ, N = m2 + (2.0f * Z + B2) * t;
        const float v2 = N * q * q;
        float Zn;
        bool done = false;
        if (!(v2 < 1.0f)) {
            lo = Z;
            Zn = 0.5f * (lo + hi);
        } else {
            const float iW2 = 1.0f - v2, rs = rsqrtf(iW2), dv2 = (-2.0f * t * (1.0f + B2 * iZ) - 2.0f * N * q) * q * q;
            const float f = Z - 1.0f - g * (Z * iW2 - D * (iW2 * rs)) + 0.5f * (B2 * (1.0f + v2) - t);
            const float df = 1.0f - g * (iW2 - Z * dv2 + 0.5f * D * dv2 * rs) + 0.5f * B2 * dv2 + t * iZ;
            if (f < 0.0f) lo = Z; else hi = Z;
            Zn = Z - f * __frcp_rn(df);
            done = fabsf(Zn - Z) <= 2.0e-4f * Z * iW2;   // (as in c2p_estimate)
            if (!done && !(Zn > lo && Zn < hi)) Zn = 0.5f * (lo + hi);
        }
        Z = Zn;
        if (done) break;
    }
    return Z;
}

static __device__ __noinline__ int c2p_loop_mhd(double g, double D, double m2, double B2, double S2, double E, double hi,
                                                double &Z)
{
    double lo = 0.0;
#pragma unroll 1
    for (int it = 0; it < 300; ++it) {
        const double iZ = __drcp_rn(Z), iZB = __drcp_rn(Z + B2), N = m2 + (2.0 * Z + B2) * S2 * iZ * iZ, v2 = N * iZB * iZB;
        double Zn;
        if (!(v2 < 1.0)) {
            lo = Z;
            Zn = 0.5 * (lo + hi);
        } else {
            const double iW2 = 1.0 - v2, rs = rsqrt(iW2), iW = iW2 * rs;
            const double p = g * (Z * iW2 - D * iW);
            const double f = Z - p + 0.5 * B2 * (1.0 + v2) - 0.5 * S2 * iZ * iZ - E;
            if (fabs(f) <= 2.0e-15 * (E + Z)) return 0;   // residual at rounding level
            const double dN = -2.0 * S2 * iZ * iZ - 2.0 * B2 * S2 * iZ * iZ * iZ;
            const double dv2 = dN * iZB * iZB - 2.0 * N * iZB * iZB * iZB;
            const double dp = g * (iW2 - Z * dv2 + 0.5 * D * dv2 * rs);
            const double df = 1.0 - dp + 0.5 * B2 * dv2 + S2 * iZ * iZ * iZ;
            if (f < 0.0) lo = Z; else hi = Z;
            Zn = Z - f * f2d_int(__frcp_rn(d2f_int(df)));   // (the slope only steers the step)
            if (!(Zn > lo && Zn < hi)) Zn = 0.5 * (lo + hi);
        }
        const bool done = fabs(Zn - Z) <= 1.0e-15 * (E + Zn);
        Z = Zn;
        if (done) return 0;
    }
    return 2;
}

__device__ __forceinline__ int cons2prim_mhd(double gam, const double U[8], double Z0, double w[8], double &Zout)
{
    const double D = U[0], E = U[4];
    const double m0 = U[1], m1 = U[2], m2_ = U[3], B0 = U[5], B1 = U[6], B2_ = U[7];
    const double m2 = m0 * m0 + m1 * m1 + m2_ * m2_;
    const double B2 = B0 * B0 + B1 * B1 + B2_ * B2_;
    const double S = m0 * B0 + m1 * B1 + m2_ * B2_;
    const double S2 = S * S;
    const double g = (gam - 1.0) / gam;
    for (int a = 0; a < 8; ++a) w[a] = 0.0;
    Zout = 0.0;
    if (!(D > 0.0) || !(E > 0.0)) return 1;
    const double hi = gam * E;
    const double Zw = (Z0 > 0.0 && Z0 < hi) ? Z0 : 0.5 * hi;
    const int k = binade(E);
    const float Ef = d2f_scaled(E, k), iE = __frcp_rn(Ef), gf = d2f_int(g), Df = d2f_scaled(D, k) * iE;
    const float B2f = d2f_scaled(B2, k) * iE, m2f = d2f_scaled(m2, 2 * k) * iE * iE, S2f = d2f_scaled(S2, 3 * k) * iE * iE * iE;
    const float Zf = c2p_estimate_mhd(gf, d2f_int(gam), Df, m2f, B2f, S2f, d2f_scaled(Zw, k) * iE);
    double Z = f2d_scaled(Zf * Ef, k);
    int st = 0;
    bool ok = false;
#pragma unroll 1
    for (int it = 0; it < 3; ++it) {   // (a second step where the estimate was poor)
        const double iZ = qrcp<double>(Z), iZB = qrcp<double>(Z + B2), t = S2 * iZ * iZ, N = m2 + (2.0 * Z + B2) * t;
        const double q2 = iZB * iZB, v2 = N * q2, iW2 = 1.0 - v2, rs = qrsq<double>(iW2), Dw = D * rs;
        const double f = (Z - E) - g * (Z * iW2 - Dw * iW2) + 0.5 * (B2 * (1.0 + v2) - t);
        const double dv2 = -2.0 * (t * (1.0 + B2 * iZ) + N * iZB) * q2;
        const double df = 1.0 - g * (iW2 - dv2 * (Z - 0.5 * Dw)) + 0.5 * B2 * dv2 + t * iZ;
        const double dZ = f * qrcp<double>(df);
        // f'' in units of E (Z = z E): v2'' = N'' q^2 - 4 N' q^3 + 6 N q^4
        const float z = d2f_scaled(Z, k) * iE, iz = __frcp_rn(z), q = __frcp_rn(z + B2f), tf = S2f * iz * iz, Nf = m2f + (2.0f * z + B2f) * tf;
        const float N1 = -2.0f * tf * (1.0f + B2f * iz), N2 = tf * iz * (4.0f + 6.0f * B2f * iz), qq = q * q;
        const float v1 = (N1 - 2.0f * Nf * q) * qq, v22 = (N2 - 4.0f * N1 * q + 6.0f * Nf * qq) * qq, sf = d2f_int(rs);
        const float p2 = gf * (-2.0f * v1 - z * v22 + 0.5f * Df * sf * (v22 + 0.5f * v1 * v1 * (sf * sf)));
        const float f2 = -p2 + 0.5f * B2f * v22 - 3.0f * tf * (iz * iz);
        const float dz = d2f_scaled(dZ, k) * iE, eta = 0.5f * f2 * dz * __frcp_rn(d2f_int(df));
        ok = fabsf(dz) <= 3.0e-6f * z * d2f_int(iW2) && fabsf(eta) <= 3.0e-6f;
        const double Zn = Z - __fma_rn(dZ, f2d_int(eta), dZ);
        if (!(d2f_scaled(Zn, k) > 0.0f) || !(fabsf(eta) <= 0.1f)) {
            ok = false;
            break;
        }
        Z = Zn;
        if (ok) break;
    }
    if (!ok) {
        Z = Zw;
        st = c2p_loop_mhd(g, D, m2, B2, S2, E, hi, Z);
    }
    const double iZ = ok ? qrcp<double>(Z) : __drcp_rn(Z), iZB = ok ? qrcp<double>(Z + B2) : __drcp_rn(Z + B2);
    const double v2 = (m2 + (2.0 * Z + B2) * S2 * iZ * iZ) * iZB * iZB;
    if (!(v2 < 1.0)) return 1;
    const double iW2 = 1.0 - v2, iW = ok ? iW2 * qrsq<double>(iW2) : sqrt(iW2);
    double vB = S * iZ;
    w[0] = D * iW;
    w[1] = (m0 + vB * B0) * iZB;
    w[2] = (m1 + vB * B1) * iZB;
    w[3] = (m2_ + vB * B2_) * iZB;
    w[4] = g * (Z * iW2 - D * iW);
    w[5] = B0; w[6] = B1; w[7] = B2_;
    Zout = Z;
    if (!(w[4] > 0.0)) return 1;
    return st;
}

// U(w), F_1(w) and V(w) (eq. RMHDdiv2, Sec. 2), generic in the number type
// so that dual numbers give directional derivatives.
template <typename T> __device__ __forceinline__ T lg(T x);
template <> __device__ __forceinline__ double lg<double>(double x) { return log(x); }
template <> __device__ __forceinline__ dual lg<dual>(dual x) { return dual(log(x.v), x.d * __drcp_rn(x.v)); }
template <> __device__ __forceinline__ fdual lg<fdual>(fdual x) { return fdual(logf(x.v), x.d * __frcp_rn(x.v)); }
template <> __device__ __forceinline__ hdual lg<hdual>(hdual x)
{
    double r = __drcp_rn(x.v);
    return hchain(x, log(x.v), r, -r * r);
}

template <typename T>
__device__ __forceinline__ void mhd_UFV(double gam, const T w[8], T U[8], T F[8], T V[8])
{
    T rho = w[0], p = w[4];
    T v2 = w[1] * w[1] + w[2] * w[2] + w[3] * w[3];
    T iW2 = 1.0 - v2;
    T W = rsq<T>(iW2);                 // (reciprocals and rsqrt: no FP64 quotient)
    T W2 = W * W;
    T vB = w[1] * w[5] + w[2] * w[6] + w[3] * w[7];
    T B2 = w[5] * w[5] + w[6] * w[6] + w[7] * w[7];
    T bb = B2 * iW2 + vB * vB;
    T rhoh = rho + (gam / (gam - 1.0)) * p;
    T pt = p + 0.5 * bb;
    T Q = rhoh * W2 + B2;
    U[0] = rho * W;
#pragma unroll
    for (int k = 0; k < 3; ++k) U[1 + k] = Q * w[1 + k] - vB * w[5 + k];
    U[4] = rhoh * W2 - pt + B2;
#pragma unroll
    for (int k = 0; k < 3; ++k) U[5 + k] = w[5 + k];
    F[0] = U[0] * w[1];
#pragma unroll
    for (int k = 0; k < 3; ++k) F[1 + k] = U[1 + k] * w[1] - w[5] * (w[5 + k] * iW2 + vB * w[1 + k]);
    F[1] = F[1] + pt;
    F[4] = U[1];
#pragma unroll
    for (int k = 0; k < 3; ++k) F[5 + k] = w[1] * w[5 + k] - w[5] * w[1 + k];
    T beta = rho * rcp<T>(p);
    T s = lg<T>(p) - gam * lg<T>(rho);
    V[0] = (gam - s) * (1.0 / (gam - 1.0)) + beta;
#pragma unroll
    for (int k = 0; k < 3; ++k) V[1 + k] = beta * W * w[1 + k];
    V[4] = -beta * W;
    const T bW = beta * iW2 * W;       // beta / W
#pragma unroll
    for (int k = 0; k < 3; ++k) V[5 + k] = bW * (w[5 + k] + W2 * w[1 + k] * vB);
}

// Images (dU, dV, dF~) of the primitive perturbation dir at w, with the
// Godunov-Powell column: dF~ = dF_1 + Phi'(V) dB_1, in the working precision R.
template <typename R>
__device__ __forceinline__ void mhd_images(double gam, const R w[8], const R dir[8], const R Pp[8], R dU[8], R dV[8],
                                           R dF[8])
{
    using D = typename DualOf<R>::type;
    D wd[8], U[8], F[8], V[8];
#pragma unroll
    for (int a = 0; a < 8; ++a) wd[a] = img_seed(w[a], dir[a]);
    mhd_UFV<D>(gam, wd, U, F, V);
#pragma unroll
    for (int a = 0; a < 8; ++a) {
        dU[a] = img_part(U[a]);
        dV[a] = img_part(V[a]);
        dF[a] = img_part(F[a]) + Pp[a] * dir[5];
    }
}

template <typename R>
__device__ __forceinline__ R dot8(const R *a, const R *b)
{
    R s = (R)0;
#pragma unroll
    for (int r = 0; r < 8; ++r) s += a[r] * b[r];
    return s;
}

// f(0) ... f(n - 1), in a rolled loop in the FP32 instances, whose kernels are
// limited by instruction fetch (the unrolled copies of these loop bodies do
// not fit the instruction cache); as the compiler chooses otherwise.
template <typename R, typename F>
__device__ __forceinline__ void each_index(int n, F &&f)
{
    if constexpr (std::is_same<R, float>::value) {
#pragma unroll 1
        for (int i = 0; i < n; ++i) f(i);
    } else {
        for (int i = 0; i < n; ++i) f(i);
    }
}

// Phi'(V) = (0, B/W^2 + v (v.B), v.B, v) (eq. Phi)
template <typename R>
__device__ __forceinline__ void mhd_phiprime(const R w[8], R P[8])
{
    R iW2 = (R)1 - (w[1] * w[1] + w[2] * w[2] + w[3] * w[3]);
    R vB = w[1] * w[5] + w[2] * w[6] + w[3] * w[7];
    P[0] = (R)0;
#pragma unroll
    for (int k = 0; k < 3; ++k) P[1 + k] = w[5 + k] * iW2 + w[1 + k] * vB;
    P[4] = vB;
#pragma unroll
    for (int k = 0; k < 3; ++k) P[5 + k] = w[1 + k];
}

// Scaled eigenvectors of the symmetrized x_1 system (Sec. 4) at the rotated
// primitive state w: lam[8] and R[8][8] (row = component, column = wave)
// with R R^T = dU/dV.  Construction (as the paper only cites formulas):
// <a, b> = dU(a).dV(b), k(a, b) = dV(a).dF~(b); the entropy wave e_rho and
// the divergence wave dB = e_1 - v_1 v have speed v_1; the other six waves
// span the <.,.> complement of y_a = e_a - projections (a = v_1, v_2, v_3,
// p, B_2, B_3) and come from cyclic Jacobi on C = L^-1 K L^-T (G = L L^T);
// clusters of speeds closer than CLUSTER_TOL get the canonical basis of
// their span (Gram-Schmidt, in index order, of the projected C-space unit
// vectors whose remaining squared norm is at least 1/8: continuous in the
// span, unlike a largest-norm choice, which switches on the exact ties of
// symmetric states).  eigen_mhd_gram builds them so; the flux kernels take the same waves
// in closed form (es_dissipation_mhd).
constexpr double MHD_CLUSTER_TOL = 1.0e-5;

// Cyclic Jacobi on the symmetric 6 x 6 C (in place: its diagonal becomes the
// eigenvalues), accumulating the rotations in Q when want_vectors.
template <typename S>
__device__ __forceinline__ void jacobi6(S C[6][6], S Q[6][6], bool want_vectors)
{
    for (int a = 0; a < 6; ++a)
        for (int b = 0; b < 6; ++b) Q[a][b] = a == b ? (S)1 : (S)0;
    // converged when the off-diagonal part is at rounding level: (1e-15)^2
    // of the diagonal in FP64, (1e-6)^2 in FP32 (the next sweep squares it)
    const S conv = sizeof(S) == 4 ? (S)1.0e-12 : (S)1.0e-30;
    for (int sweep = 0; sweep < 50; ++sweep) {
        S off = (S)0, dg = (S)0;
        for (int a = 0; a < 6; ++a) {
            dg += C[a][a] * C[a][a];
            for (int b = a + 1; b < 6; ++b) off += C[a][b] * C[a][b];
        }
        if (off <= conv * dg) break;
        // The rotation loops stay rolled: fully unrolled, this sweep came out
        // of nvcc 13.0 -O3 (sm_103a) as a non-similarity transform (wrong
        // eigenvalues; the host build and the -G build of the same source are
        // right), so unrolling is disabled here.
#pragma unroll 1
        for (int p = 0; p < 5; ++p)
#pragma unroll 1
            for (int q = p + 1; q < 6; ++q) {
                if (C[p][q] == (S)0) continue;
                // (reciprocals for the rotation's quotients: FP64 divisions
                // cost ~15 FP64-pipe instructions each on this GPU).  A tiny
                // C_pq can have an infinite reciprocal: equal diagonals then
                // take theta = 0 (as the quotient 0 / (2 C_pq) does), unequal
                // ones theta = +-inf, hence t = 0 (no rotation)
                const S diff = C[q][q] - C[p][p];
                S theta = diff == (S)0 ? (S)0 : diff * ((S)0.5 * rcp<S>(C[p][q]));
                S t = (theta >= (S)0 ? (S)1 : (S)-1) * rcp<S>(fab<S>(theta) + sq_rt<S>(theta * theta + (S)1));
                S cs = rsq<S>(t * t + (S)1), sn = t * cs;
#pragma unroll 1
                for (int k = 0; k < 6; ++k) {
                    S ckp = C[k][p], ckq = C[k][q];
                    C[k][p] = cs * ckp - sn * ckq;
                    C[k][q] = sn * ckp + cs * ckq;
                }
#pragma unroll 1
                for (int k = 0; k < 6; ++k) {
                    S cpk = C[p][k], cqk = C[q][k];
                    C[p][k] = cs * cpk - sn * cqk;
                    C[q][k] = sn * cpk + cs * cqk;
                }
                if (want_vectors)
#pragma unroll 1
                    for (int k = 0; k < 6; ++k) {
                        S qkp = Q[k][p], qkq = Q[k][q];
                        Q[k][p] = cs * qkp - sn * qkq;
                        Q[k][q] = sn * qkp + cs * qkq;
                    }
            }
    }
}

template <typename R>
static __device__ __noinline__ void eigen_mhd_gram(double gam, const R w[8], R lam[8], R Rv[8][8], bool want_vectors)
{
    R Pp[8];
    mhd_phiprime(w, Pp);
    const R v1 = w[1];
    R a_rho[8] = {(R)1, (R)0, (R)0, (R)0, (R)0, (R)0, (R)0, (R)0};
    R a_div[8] = {(R)0, (R)0, (R)0, (R)0, (R)0, (R)1 - v1 * v1, -v1 * w[2], -v1 * w[3]};
    R Ur[8], Vr[8], Fr[8], Ud[8], Vd[8], Fd[8];
    mhd_images(gam, w, a_rho, Pp, Ur, Vr, Fr);
    mhd_images(gam, w, a_div, Pp, Ud, Vd, Fd);
    const R n_rho = dot8(Ur, Vr), n_div = dot8(Ud, Vd);
    const R in_rho = rcp<R>(n_rho), in_div = rcp<R>(n_div);
    const int comp[6] = {1, 2, 3, 4, 6, 7};
    R Uy[6][8], Vy[6][8], Fy[6][8];
    each_index<R>(6, [&](int a) {
        R e[8] = {(R)0, (R)0, (R)0, (R)0, (R)0, (R)0, (R)0, (R)0};
        e[comp[a]] = (R)1;
        R Ue[8], Ve[8], Fe[8];
        mhd_images(gam, w, e, Pp, Ue, Ve, Fe);
        R cr = dot8(Ue, Vr) * in_rho, cd = dot8(Ue, Vd) * in_div;
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            Uy[a][r] = Ue[r] - cr * Ur[r] - cd * Ud[r];
            Vy[a][r] = Ve[r] - cr * Vr[r] - cd * Vd[r];
            Fy[a][r] = Fe[r] - cr * Fr[r] - cd * Fd[r];
        }
        if constexpr (std::is_same<R, float>::value) {
            // FP32: scale y_a to unit <y_a, y_a> (the Gram diagonal spans
            // many decades at large W); C = L^-1 K L^-T is unchanged by it
            R sa = rsq<R>(dot8(Uy[a], Vy[a]));
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                Uy[a][r] *= sa;
                Vy[a][r] *= sa;
                Fy[a][r] *= sa;
            }
        }
    });
    R Gm[6][6], C[6][6];
    each_index<R>(6, [&](int a) {
        each_index<R>(a + 1, [&](int b) {
            R g = (R)0.5 * (dot8(Uy[a], Vy[b]) + dot8(Uy[b], Vy[a]));
            R k = (R)0.5 * (dot8(Vy[a], Fy[b]) + dot8(Vy[b], Fy[a]));
            Gm[a][b] = Gm[b][a] = g;
            C[a][b] = C[b][a] = k;
        });
    });
    // Cholesky G = L L^T (lower triangle of Gm), with the reciprocals of
    // its diagonal (idg) serving every division of the factor and the solves
    R idg[6];
    for (int j = 0; j < 6; ++j) {
        R d = Gm[j][j];
        for (int k = 0; k < j; ++k) d -= Gm[j][k] * Gm[j][k];
        if constexpr (std::is_same<R, float>::value)
            if (!(d > (R)1.0e-12)) d = (R)1.0e-12;   // FP32: keep the factor finite
        Gm[j][j] = sq_rt<R>(d);
        idg[j] = rcp<R>(Gm[j][j]);
        for (int i = j + 1; i < 6; ++i) {
            R s = Gm[i][j];
            for (int k = 0; k < j; ++k) s -= Gm[i][k] * Gm[j][k];
            Gm[i][j] = s * idg[j];
        }
    }
    // C <- L^-1 K L^-T (column solves, then row solves)
    for (int c = 0; c < 6; ++c)
        for (int i = 0; i < 6; ++i) {
            R s = C[i][c];
            for (int k = 0; k < i; ++k) s -= Gm[i][k] * C[k][c];
            C[i][c] = s * idg[i];
        }
    for (int r = 0; r < 6; ++r)
        for (int i = 0; i < 6; ++i) {
            R s = C[r][i];
            for (int k = 0; k < i; ++k) s -= Gm[i][k] * C[r][k];
            C[r][i] = s * idg[i];
        }
    for (int a = 0; a < 6; ++a)
        for (int b = 0; b < a; ++b) C[a][b] = C[b][a] = (R)0.5 * (C[a][b] + C[b][a]);
    int ord[6] = {0, 1, 2, 3, 4, 5};
    R E6[6][6];
    if constexpr (std::is_same<R, dual>::value) {
        // Adjoint tangent: Jacobi on the values; first-order perturbation
        // theory for the tangent.  With M = Q^T C' Q (C' = C.d), an eigenvalue
        // moves by M_ii and eigenvector i by sum_j M_ji / (lam_i - lam_j) e_j
        // over the j outside i's cluster: inside a cluster only the span is
        // defined, and the canonical basis below is a function of the span.
        double Cv[6][6], Qv[6][6], M[6][6];
        for (int i = 0; i < 6; ++i)
            for (int j = 0; j < 6; ++j) Cv[i][j] = C[i][j].v;
        jacobi6<double>(Cv, Qv, true);
        for (int i = 0; i < 6; ++i)
            for (int j = 0; j < 6; ++j) {
                double acc = 0.0;
                for (int k = 0; k < 6; ++k)
                    for (int l = 0; l < 6; ++l) acc += Qv[k][i] * C[k][l].d * Qv[l][j];
                M[i][j] = acc;
            }
        for (int a = 0; a < 6; ++a)
            for (int b = a + 1; b < 6; ++b)
                if (Cv[ord[b]][ord[b]] < Cv[ord[a]][ord[a]]) { int t = ord[a]; ord[a] = ord[b]; ord[b] = t; }
        int cl[6];   // cluster id of each sorted wave
        cl[0] = 0;
        for (int m = 1; m < 6; ++m)
            cl[m] = cl[m - 1] + (Cv[ord[m]][ord[m]] - Cv[ord[m - 1]][ord[m - 1]] < MHD_CLUSTER_TOL ? 0 : 1);
        for (int m = 0; m < 6; ++m) {
            const int i = ord[m];
            const double li = Cv[i][i];
            lam[2 + m] = dual(li, M[i][i]);
            if (!want_vectors) continue;
            for (int r = 0; r < 6; ++r) {
                double t = 0.0;
                for (int n = 0; n < 6; ++n) {
                    if (cl[n] == cl[m]) continue;
                    const int j = ord[n];
                    t += M[j][i] / (li - Cv[j][j]) * Qv[r][j];
                }
                E6[r][m] = dual(Qv[r][i], t);
            }
        }
        lam[0] = v1;
        lam[1] = v1;
        if (!want_vectors) return;
    } else {
        R Q[6][6];
        jacobi6<R>(C, Q, want_vectors);
        for (int a = 0; a < 6; ++a)
            for (int b = a + 1; b < 6; ++b)
                if (C[ord[b]][ord[b]] < C[ord[a]][ord[a]]) { int t = ord[a]; ord[a] = ord[b]; ord[b] = t; }
        lam[0] = v1;
        lam[1] = v1;
        for (int m = 0; m < 6; ++m) lam[2 + m] = C[ord[m]][ord[m]];
        if (!want_vectors) return;
        for (int m = 0; m < 6; ++m)
            for (int r = 0; r < 6; ++r) E6[r][m] = Q[r][ord[m]];
    }
    int start = 0;
    while (start < 6) {
        int end = start + 1;
        while (end < 6 && val(lam[2 + end]) - val(lam[1 + end]) < MHD_CLUSTER_TOL) ++end;
        const int k = end - start;
        if (k > 1) {
            // Gram-Schmidt in index order of the C-space unit vectors projected
            // on the cluster's span, taking those with remaining squared norm
            // >= 1/8 (k of them always are: the six squared norms sum to k)
            R z[6][6], basis[6][6];
            for (int i = 0; i < 6; ++i)
                for (int c = 0; c < k; ++c) z[i][c] = E6[i][start + c];
            int nt = 0;
            for (int i = 0; i < 6 && nt < k; ++i) {
                R n2 = (R)0;
                for (int c = 0; c < k; ++c) n2 += z[i][c] * z[i][c];
                if (!(val(n2) >= 0.125)) continue;
                R inr = (R)1 / sq_rt<R>(n2);
                for (int c = 0; c < k; ++c) basis[nt][c] = z[i][c] * inr;
                for (int ii = i + 1; ii < 6; ++ii) {
                    R pr = (R)0;
                    for (int c = 0; c < k; ++c) pr += z[ii][c] * basis[nt][c];
                    for (int c = 0; c < k; ++c) z[ii][c] -= pr * basis[nt][c];
                }
                ++nt;
            }
            if (nt < k) {   // only for non-finite input: keep the Jacobi basis
                start = end;
                continue;
            }
            R nE[6][6];
            for (int t = 0; t < k; ++t)
                for (int r = 0; r < 6; ++r) {
                    R acc = (R)0;
                    for (int c = 0; c < k; ++c) acc += E6[r][start + c] * basis[t][c];
                    nE[r][t] = acc;
                }
            for (int t = 0; t < k; ++t)
                for (int r = 0; r < 6; ++r) E6[r][start + t] = nE[r][t];
        }
        start = end;
    }
    const R srho = rsq<R>(n_rho), sdiv = rsq<R>(n_div);
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        Rv[r][0] = Ur[r] * srho;
        Rv[r][1] = Ud[r] * sdiv;
    }
    each_index<R>(6, [&](int m) {
        R s[6];
        for (int i = 5; i >= 0; --i) {
            R acc = E6[i][m];
            for (int k = i + 1; k < 6; ++k) acc -= Gm[k][i] * s[k];
            s[i] = acc * idg[i];
        }
        for (int r = 0; r < 8; ++r) {
            R acc = (R)0;
            for (int a = 0; a < 6; ++a) acc += s[a] * Uy[a][r];
            Rv[r][2 + m] = acc;
        }
    });
}

}  // namespace esmm

#include "esmm_mhd_waves.cuh"

namespace esmm {

// the smallest and largest speed (the fast waves) at the rotated state w: the
// CFL radius needs no vectors
template <typename R>
static __device__ __noinline__ void mhd_speed_range(double gam, const R w[8], R &lo, R &hi)
{
    MhdBase<R> s;
    mhd_base<R>((R)gam, (R)(gam / (gam - 1.0)), w, s);
    if (!mhd_in_range<R>(s)) {
        R lam[8], Rm[8][8];
        eigen_mhd_gram<R>(gam, w, lam, Rm, false);
        lo = lam[2];
        hi = lam[7];
        return;
    }
    MhdCoef<R> kc;
    mhd_coef<R>(s, kc);
    R tA, ts, tf;
    mhd_side<R>(s, kc, 1, false, tA, ts, tf);
    lo = s.v1 - tf * s.iW;
    mhd_side<R>(s, kc, -1, false, tA, ts, tf);
    hi = s.v1 + tf * s.iW;
}

// The canonical basis (see eigen_mhd_gram) of a cluster of two waves a, b of one side, an
// Alfven and a magnetosonic one: they are orthogonal whatever their speeds (s is normal to
// t, k and b), so a rotation of the two columns is all that is needed, and its first
// vector is the first row (E[i][a], E[i][b]) of E = L^T S whose squared norm is at least
// 1/8; the second is the complement.  Row i takes the directions e_0 .. e_i alone, and
// e_0 or e_1 (v_1, v_2) nearly always decides: e_{v_k} in closed form,
//   du = (W u_k, e_k + u_k u) (times W), db from B = const,  dV = beta (0, du, -du^0, db),
// with <e_i, a> = dV(e_i).R_a, and <e_i, e_j> from the bilinear form X^0.  Returns false
// where neither row decides.  (~150 operations, against ~1,000 with the whole Gram
// matrix: a rotor's ambient field along x_1 leaves clusters in half the interfaces
// of that sweep.)  Rv: rows dU of the waves, rows 0 and 1 the entropy and divergence waves.
template <typename R>
__device__ __forceinline__ bool mhd_turn_pair(const MhdBase<R> &s, const R B[3], R Rv[8][8], int a)
{
    R du[2][4], db[2][4], P[2], c, sn;
    R Ea = (R)0, Eb = (R)0, i0 = (R)0, f0r = (R)0, f0d = (R)0;
    bool ok = false;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        if (ok) break;
        const R uk = s.u[1 + i];
        du[i][0] = s.W * uk;
#pragma unroll
        for (int k = 1; k < 4; ++k) du[i][k] = (k == 1 + i ? (R)1 : (R)0) + s.u[k] * uk;
        db[i][0] = du[i][1] * B[0] + du[i][2] * B[1] + du[i][3] * B[2];
#pragma unroll
        for (int k = 1; k < 4; ++k) db[i][k] = (db[i][0] * s.u[k] + s.b[0] * du[i][k] - s.b[k] * du[i][0]) * s.iW;
        P[i] = mdot<R>(s.b, db[i]);
        R f[4];   // <e_i, .> with the entropy, the divergence wave, a and b, over beta
#pragma unroll
        for (int n = 0; n < 4; ++n) {
            const R *r = n < 2 ? Rv[n] : Rv[a + n - 2];
            f[n] = du[i][1] * r[1] + du[i][2] * r[2] + du[i][3] * r[3] - du[i][0] * r[4] + db[i][1] * r[5] + db[i][2] * r[6] +
                   db[i][3] * r[7];
        }
        // Gram entries over beta
        const R gii = s.W * (s.e * mdot<R>(du[i], du[i]) + mdot<R>(db[i], db[i])) +
                      (R)2 * (du[i][0] * P[i] - s.b[0] * mdot<R>(db[i], du[i])) - s.beta * (f[0] * f[0] + f[1] * f[1]);
        R ea = f[2], eb = f[3], d = gii;
        if (i == 0) {
            f0r = f[0];
            f0d = f[1];
        } else {
            const R g10 = s.W * (s.e * mdot<R>(du[0], du[1]) + mdot<R>(db[0], db[1])) + du[0][0] * P[1] + du[1][0] * P[0] -
                          s.b[0] * (mdot<R>(db[0], du[1]) + mdot<R>(db[1], du[0])) - s.beta * (f0r * f[0] + f0d * f[1]);
            const R l = g10 * i0;   // L_10 over L_00, times sqrt(g00)
            d -= l * g10;
            ea -= l * Ea;
            eb -= l * Eb;
        }
        // |row|^2 = beta (ea^2 + eb^2) / d
        const R n2 = ea * ea + eb * eb;
        if (to_f32(s.beta * n2) >= 0.125f * to_f32(d)) {
            const R inr = qrsq<R>(n2);
            c = ea * inr;
            sn = eb * inr;
            ok = true;
        }
        Ea = ea;
        Eb = eb;
        i0 = qrcp<R>(gii);
    }
    if (!ok) return false;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        const R x = Rv[a][r], y = Rv[a + 1][r];
        Rv[a][r] = c * x + sn * y;
        Rv[a + 1][r] = c * y - sn * x;
    }
    return true;
}

// The canonical basis of every cluster among the six waves (bit m of near: waves m and m + 1
// are in one), whose rows dU of Rv it replaces: with the directions e_i = v_1, v_2, v_3 (times
// 1/W), p, B_2, B_3 in closed form (as in mhd_turn_pair; p: du = db = 0, dV = -(beta/p)
// (1 + 1/((Gamma-1) beta), u, -W, b); B_k: db = e_k/W + u_k (1, u/W), dV = beta (0, 0, 0, db)), their
// Gram matrix G = L L^T off the entropy and divergence waves and S[i][m] the wave m's
// coefficients in the e_i, the waves in C-space are E = L^T S; each cluster is orthonormalized there (twice: its waves
// may be oblique at rounding level over their gap) and takes the Gram-Schmidt of the
// unit vectors projected on its span, both as a matrix on its rows of Rv.  ~1,000
// FP64 instructions, against ~3,500 with the images on dual numbers and the waves formed
// anew; four waves of one speed are the rule where B_n = 0.  Measured: the untapered 512^2
// rotor step 16.1 -> 13.4 ms, mixed 2.36 -> 1.94 ms, a 64^3 blast step at rest 29.4 -> 23.2 ms,
// a 64^3 step of gas without a field 36.7 -> 27.6 ms.
template <typename R>
static __device__ __noinline__ void mhd_turn_clusters(const MhdBase<R> &s, R ig, const R B[3], R S[6][6], R Rv[8][8],
                                                          int near)
{
    R du[3][4], db[5][4], P[5], f0[6], f1[6], G[6][6], E[6][6];
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        if (k < 3) {
            const R uk = s.u[1 + k];
            du[k][0] = s.W * uk;
#pragma unroll
            for (int q = 1; q < 4; ++q) du[k][q] = (q == 1 + k ? (R)1 : (R)0) + s.u[q] * uk;
            db[k][0] = du[k][1] * B[0] + du[k][2] * B[1] + du[k][3] * B[2];
#pragma unroll
            for (int q = 1; q < 4; ++q) db[k][q] = (db[k][0] * s.u[q] + s.b[0] * du[k][q] - s.b[q] * du[k][0]) * s.iW;
        } else {   // B_2, B_3
            const R uk = s.u[k - 1];
            db[k][0] = uk;
#pragma unroll
            for (int q = 1; q < 4; ++q) db[k][q] = ((q == k - 1 ? (R)1 : (R)0) + uk * s.u[q]) * s.iW;
        }
        P[k] = mdot<R>(s.b, db[k]);
    }
    // <e_i, .> over beta with the entropy and the divergence wave (index of db: v 0..2, B 3,
    // 4; of f0: v 0..2, p 3, B 4, 5)
    const R cp = (R)1 + ig * rcp<R>(s.beta);
#pragma unroll
    for (int m = 0; m < 2; ++m) {
        const R *r = Rv[m];
        R *f = m == 0 ? f0 : f1;
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            R acc = db[k][1] * r[5] + db[k][2] * r[6] + db[k][3] * r[7];
            if (k < 3) acc += du[k][1] * r[1] + du[k][2] * r[2] + du[k][3] * r[3] - du[k][0] * r[4];
            f[k < 3 ? k : k + 1] = acc;
        }
        f[3] = -s.ip * (cp * r[0] + s.u[1] * r[1] + s.u[2] * r[2] + s.u[3] * r[3] - s.W * r[4] + s.b[1] * r[5] + s.b[2] * r[6] +
                        s.b[3] * r[7]);
    }
    // Gram entries over beta, scaled to a unit diagonal (E is unchanged by that)
#pragma unroll
    for (int a = 0; a < 5; ++a)
#pragma unroll
        for (int b = 0; b <= a; ++b) {
            R g = s.W * mdot<R>(db[a], db[b]);
            if (a < 3) {
                g += s.W * (s.e * mdot<R>(du[a], du[b])) + du[a][0] * P[b] + du[b][0] * P[a] -
                     s.b[0] * (mdot<R>(db[a], du[b]) + mdot<R>(db[b], du[a]));
            } else if (b < 3) {
                g += du[b][0] * P[a] - s.b[0] * mdot<R>(db[a], du[b]);
            }
            G[a < 3 ? a : a + 1][b < 3 ? b : b + 1] = g;
        }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        G[3][k] = du[k][0];
        if (k < 2) G[4 + k][3] = (R)0;
    }
    G[3][3] = s.W * s.ip * ig;   // (Gamma/(Gamma-1) - 1 = 1/(Gamma-1))
    R sc[6];
#pragma unroll
    for (int a = 0; a < 6; ++a) {
#pragma unroll
        for (int b = 0; b <= a; ++b) G[a][b] -= s.beta * (f0[a] * f0[b] + f1[a] * f1[b]);
        sc[a] = rsq<R>(G[a][a]);
    }
#pragma unroll
    for (int a = 0; a < 6; ++a)
#pragma unroll
        for (int b = 0; b <= a; ++b) G[a][b] *= sc[a] * sc[b];
#pragma unroll 1
    for (int j = 0; j < 6; ++j) {
        R d = G[j][j];
        for (int k = 0; k < j; ++k) d -= G[j][k] * G[j][k];
        if constexpr (sizeof(R) == 4)
            if (!(d > (R)1.0e-12)) d = (R)1.0e-12;   // FP32: keep the factor finite
        const R idg = rsq<R>(d);
        G[j][j] = d * idg;
        for (int i = j + 1; i < 6; ++i) {
            R t = G[i][j];
            for (int k = 0; k < j; ++k) t -= G[i][k] * G[j][k];
            G[i][j] = t * idg;
        }
        sc[j] = rcp<R>(sc[j]);
        for (int m = 0; m < 6; ++m) S[j][m] *= sc[j];
    }
#pragma unroll 1
    for (int i = 0; i < 6; ++i)   // E over sqrt(beta): its columns are normalized below
        for (int m = 0; m < 6; ++m) {
            R t = G[i][i] * S[i][m];
            for (int j = i + 1; j < 6; ++j) t += G[j][i] * S[j][m];
            E[i][m] = t;
        }
    const R isb = rsq<R>(s.beta);
    int start = 0;
#pragma unroll 1
    while (start < 6) {
        int end = start + 1;
        while (end < 6 && (near >> (end - 1) & 1)) ++end;
        const int k = end - start;
        if (k > 1) {
            R M[6][6], basis[6][6], z[6][6];   // M: the orthonormal members (columns) from the waves
            for (int c = 0; c < k; ++c) {
                for (int q = 0; q < k; ++q) M[q][c] = q == c ? isb : (R)0;
                for (int pass = 0; pass < 2; ++pass)
                    for (int b = 0; b < c; ++b) {
                        R pr = (R)0;
                        for (int i = 0; i < 6; ++i) pr += E[i][start + b] * E[i][start + c];
                        for (int i = 0; i < 6; ++i) E[i][start + c] -= pr * E[i][start + b];
                        for (int q = 0; q < k; ++q) M[q][c] -= pr * M[q][b];
                    }
                R n2 = (R)0;
                for (int i = 0; i < 6; ++i) n2 += E[i][start + c] * E[i][start + c];
                const R inr = rsq<R>(n2);
                for (int i = 0; i < 6; ++i) E[i][start + c] *= inr;
                for (int q = 0; q < k; ++q) M[q][c] *= inr;
            }
            for (int i = 0; i < 6; ++i)
                for (int c = 0; c < k; ++c) z[i][c] = E[i][start + c];
            int nt = 0;
            for (int i = 0; i < 6 && nt < k; ++i) {
                R n2 = (R)0;
                for (int c = 0; c < k; ++c) n2 += z[i][c] * z[i][c];
                if (!(n2 >= (R)0.125)) continue;
                const R inr = rsq<R>(n2);
                for (int c = 0; c < k; ++c) basis[nt][c] = z[i][c] * inr;
                for (int ii = i + 1; ii < 6; ++ii) {
                    R pr = (R)0;
                    for (int c = 0; c < k; ++c) pr += z[ii][c] * basis[nt][c];
                    for (int c = 0; c < k; ++c) z[ii][c] -= pr * basis[nt][c];
                }
                ++nt;
            }
            if (nt == k) {   // (less: non-finite input)
                R T[6][6];   // canonical member t = sum_q T[t][q] wave q
                for (int t = 0; t < k; ++t)
                    for (int q = 0; q < k; ++q) {
                        R acc = (R)0;
                        for (int c = 0; c < k; ++c) acc += M[q][c] * basis[t][c];
                        T[t][q] = acc;
                    }
                for (int r = 0; r < 8; ++r) {
                    R o[6];
                    for (int t = 0; t < k; ++t) {
                        R acc = (R)0;
                        for (int q = 0; q < k; ++q) acc += T[t][q] * Rv[2 + start + q][r];
                        o[t] = acc;
                    }
                    for (int t = 0; t < k; ++t) Rv[2 + start + t][r] = o[t];
                }
            }
        }
        start = end;
    }
}

// The scaled eigenvectors of one interface in its rotated frame (first axis along the
// normal; rows of Rv, one per wave) at the interface state rho, p = 1/ip, spatial
// 4-velocity us, field Bs, and the smallest and largest speed.  Clusters of two
// waves of one side are turned by mhd_turn_pair, others by mhd_turn_clusters; states outside
// the closed form's range, and where it finds no positive norm, take eigen_mhd_gram.
template <typename R>
__device__ __forceinline__ void mhd_scaled_waves(const Phys &ph, R rho, R p, R ip, const R us[3], const R Bs[3], R &lo, R &hi,
                                                 R Rv[8][8])
{
    const R gg = (R)(ph.gamma * ph.gm1i);
    MhdBase<R> s;
    const R W2 = (R)1 + (us[0] * us[0] + us[1] * us[1] + us[2] * us[2]), iW = qrsq<R>(W2);
    mhd_base_u<R>((R)ph.gamma, gg, rho, p, ip, W2 * iW, iW, us, Bs, s);
    bool whole = !mhd_in_range<R>(s);
    if (!whole) {
        MhdSix<R> x;
        R l6[6];
        mhd_six<R>(s, x, l6);
        lo = l6[0];
        hi = l6[5];
        int near = 0;   // bit m: waves m and m + 1 in one cluster
#pragma unroll
        for (int m = 0; m < 5; ++m) near |= (int)mhd_close<R>(l6[m], l6[m + 1]) << m;
        R S[6][6];
        mhd_entropy_dU<R>(s, (R)ph.igg, Rv[0]);
        mhd_divergence_dU<R>(s, Rv[1]);
#pragma unroll 1
        for (int m = 0; m < 6; ++m) {
            MhdWave<R> q;
            whole = !mhd_six_wave<R, false>(s, x, gg, m, q, Rv[2 + m]) || whole;
            if (near) {
                const R *r = Rv[2 + m], ga = -s.v1 * r[5] * qrcp<R>((R)1 - s.v1 * s.v1) * s.iW, d0 = q.u[0] * s.iW;
                for (int k = 0; k < 3; ++k) S[k][m] = q.u[1 + k] - s.u[1 + k] * d0;
                S[3][m] = q.p;
                S[4][m] = r[6] - ga * s.u[2];
                S[5][m] = r[7] - ga * s.u[3];
            }
        }
        if (near) {
            // pairs of one side (not the slow waves of both, nor three and more); a pair turned
            // here is done: S describes the waves before it
            int left = near;
            if ((near & 4) == 0 && (near & (near >> 1)) == 0)
#pragma unroll 1
                for (int m = 0; m < 5; ++m)
                    if ((near >> m & 1) && mhd_turn_pair<R>(s, Bs, Rv, 2 + m)) left &= ~(1 << m);
            if (left) mhd_turn_clusters<R>(s, (R)ph.gm1i, Bs, S, Rv, left);
        }
    }
    if (whole) {
        R lam[8], Rc[8][8];
        const R w[8] = {rho, us[0] * s.iW, us[1] * s.iW, us[2] * s.iW, p, Bs[0], Bs[1], Bs[2]};
        eigen_mhd_gram<R>(ph.gamma, w, lam, Rc, true);
        lo = lam[2];
        hi = lam[7];
        for (int m = 0; m < 8; ++m)
            for (int r = 0; r < 8; ++r) Rv[m][r] = Rc[r][m];
    }
}

// The ES dissipation of one interface in its rotated frame (first axis along the
// normal): with the interface state rho = {{rho}}^ln, u = {{u}}, p = 1/ip, B = {{B}}
// and the scaled eigenvectors R, d = lambda^/2 R Y <<R^T V>>, lambda^ the largest |jt + Lk
// lambda_m| (reached by a fast wave).  rotV(k, V) gives the rotated entropy variables of the
// stencil's node k.  The dissipation depends on differences of V alone, so those are
// projected (w of them), and the wave's edge jump comes from them (weno5_jump); the
// switch's tolerance is formed in FP32 from |R| and |V| (jump_sign).
template <typename R, int WW, typename ROTV>
__device__ __forceinline__ void es_dissipation_mhd(const Phys &ph, R rho, R p, R ip, const R us[3], const R Bs[3], R Lk,
                                                   R jt, ROTV rotV, R d[8])
{
    constexpr int OFF = (WW - 1) / 2;
    R lo, hi, Rv[8][8];   // (a row per wave)
    mhd_scaled_waves<R>(ph, rho, p, ip, us, Bs, lo, hi, Rv);
    R D[WW][8], Vo[8];   // (Vo: the left node's, for jumps that FP32 leaves open)
    float aT[8];
    {
        R V[2][8];
        rotV(0, V[0]);
#pragma unroll
        for (int k = 0; k < WW; ++k) {
            R *va = V[k & 1], *vb = V[(k + 1) & 1];
            rotV(k + 1, vb);
#pragma unroll
            for (int a = 0; a < 8; ++a) {
                if (k == OFF) {
                    aT[a] = fabsf(to_f32(va[a])) + fabsf(to_f32(vb[a]));
                    Vo[a] = va[a];
                }
                D[k][a] = sub_<R>(vb[a], va[a]);
            }
        }
    }
    jump_terms<R, 8>(aT);
#pragma unroll
    for (int a = 0; a < 8; ++a) d[a] = (R)0;
#pragma unroll 1
    for (int m = 0; m < 8; ++m) {
        R r[8];
#pragma unroll
        for (int a = 0; a < 8; ++a) r[a] = Rv[m][a];
        R Dt[WW];
#pragma unroll
        for (int k = 0; k < WW; ++k) {
            R acc = r[0] * D[k][0];
#pragma unroll
            for (int a = 1; a < 8; ++a) acc += r[a] * D[k][a];
            Dt[k] = acc;
        }
        float scale = 0.0f;
#pragma unroll
        for (int a = 0; a < 8; ++a) scale += fabsf(to_f32(r[a])) * aT[a];
        R jw;
        if constexpr (WW == 5) jw = weno5_jump<R>(Dt[0], Dt[1], Dt[2], Dt[3], Dt[4], (R)(4.0 * ph.eps));
        else jw = weno3_jump<R>(Dt[0], Dt[1], Dt[2], (R)ph.eps);
        const R jump = Dt[OFF];
        int sj = jump_sign(jump, ph.sign_tol, scale);
        if constexpr (std::is_same<R, double>::value)
            if (sj == JUMP_UNSURE) {
                double s64 = 0.0;
#pragma unroll
                for (int a = 0; a < 8; ++a) s64 += fabs(r[a]) * (fabs(Vo[a]) + fabs(Vo[a] + D[OFF][a]));
                sj = jump_sign64(jump, ph.sign_tol, s64);
            }
        const R z = sgn_d(jw) == sj ? jw : (R)0;
#pragma unroll
        for (int a = 0; a < 8; ++a) d[a] += r[a] * z;
    }
    const R hl = (R)0.5 * vmax(fab<R>(jt + Lk * lo), fab<R>(jt + Lk * hi));
#pragma unroll
    for (int a = 0; a < 8; ++a) d[a] *= hl;
}

// ---------------------------------------------------------------------------
// Node values of one two-point flux argument: the log-mean arguments (in the mixed
// form FP32 with the rest of the FP64 value) and the rest in the working precision R.
template <typename R>
struct NodeMT {
    LmV<R> rho, beta;
    R W, u[3], B[3];
};
using NodeM = NodeMT<double>;

// an FP64 value in R (the conversion off the FP64 pipe)
template <typename R> __device__ __forceinline__ R in_w(double x);
template <> __device__ __forceinline__ double in_w<double>(double x) { return x; }
template <> __device__ __forceinline__ float in_w<float>(double x) { return d2f_int(x); }

// the arrays of the flux arguments: FP64 node data, or its FP32 copies
template <typename R> struct NodeIx;
template <> struct NodeIx<double> {
    enum { RHO = Q_RHO, BETA = Q_BETA, LNR = Q_LNR, LNB = Q_LNB, W = Q_W, U0 = Q_UX, U1 = Q_UY, U2 = QM_UZ,
           B0 = QM_B1, B1 = QM_B2, B2 = QM_B3 };
};
template <> struct NodeIx<float> {
    enum { RHO = QM32_R, BETA = QM32_B, LNR = QM32_LNR, LNB = QM32_LNB, W = QM32_W, U0 = QM32_U0, U1 = QM32_U1,
           U2 = QM32_U2, B0 = QM32_B0, B1 = QM32_B1, B2 = QM32_B2 };
};

// (v: the arrays of R)
template <typename R = double>
__device__ __forceinline__ NodeMT<R> load_node_m(const R *__restrict__ v, long long P, long long c)
{
    using I = NodeIx<R>;
    NodeMT<R> n;
    n.rho.v = v[I::RHO * P + c];
    n.rho.l = v[I::LNR * P + c];
    n.beta.v = v[I::BETA * P + c];
    n.beta.l = v[I::LNB * P + c];
    if constexpr (std::is_same<R, float>::value) {
        n.rho.lo = v[QM32_RLO * P + c];
        n.beta.lo = v[QM32_BLO * P + c];
    }
    n.W = v[I::W * P + c];
    n.u[0] = v[I::U0 * P + c];
    n.u[1] = v[I::U1 * P + c];
    n.u[2] = v[I::U2 * P + c];
    n.B[0] = v[I::B0 * P + c];
    n.B[1] = v[I::B1 * P + c];
    n.B[2] = v[I::B2 * P + c];
    return n;
}

// Curvilinear two-point EC flux (Sec. 3.1) of one node pair:
//   out = mt U~ + sum_{j<NJ} m_j F~_j with the averaged metrics mt, m.
// U~: the paper's U~^RMHD with R_1 summed over three components and its
// magnetic term 1/2 {{W (b^k)^2}}; F~_j: coefficient matching with exact
// product-rule expansions, including the -{{B_j}}[[Phi]] term.  Here
// b = (B + (u.B) u)/W, b^0 = u.B, c = W b^0, v = u/W.  F~_j enters only as m.F~ and
// is linear in its direction, so it is taken once along m (u_n = m.u, B_n = m.B): the
// cost does not grow with NJ.
template <int NJ, typename R>
__device__ __forceinline__ void ec_pair_mhd(const NodeMT<R> &L, const NodeMT<R> &Rn, R gm1inv, double thr, R mt,
                                            const R m[3], R out[8])
{
    R rln, irln, bln, ibln;
    logmean2<R>(L.rho, Rn.rho, thr, rln, irln);
    logmean2<R>(L.beta, Rn.beta, thr, bln, ibln);
    const R half = (R)0.5;
    // per node: b^0, 1/W, b, b.b (spatial), u_n, B_n; sums over the two nodes
    R b[3] = {(R)0, (R)0, (R)0}, bsq = (R)0, Wbsq = (R)0, c = (R)0, b0m = (R)0, Wb0 = (R)0, Sn = (R)0, vn = (R)0,
      un = (R)0, Bn = (R)0;
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        const NodeMT<R> &n = x == 0 ? L : Rn;
        const R b0 = n.u[0] * n.B[0] + n.u[1] * n.B[1] + n.u[2] * n.B[2], iWx = qrcp<R>(n.W);
        R bk[3], ux = m[0] * n.u[0], Bx = m[0] * n.B[0];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            bk[k] = (n.B[k] + b0 * n.u[k]) * iWx;
            b[k] += bk[k];
            if (k > 0 && k < NJ) {
                ux += m[k] * n.u[k];
                Bx += m[k] * n.B[k];
            }
        }
        const R bb = bk[0] * bk[0] + bk[1] * bk[1] + bk[2] * bk[2], W0 = n.W * b0;
        bsq += bb;
        Wbsq += n.W * bb;
        c += W0;
        b0m += b0;
        Wb0 += W0 * b0;
        Sn += ux * (bb - b0 * b0);
        vn += ux * iWx;
        un += ux;
        Bn += Bx;
    }
    const R rm = half * (L.rho.v + Rn.rho.v), be = half * (L.beta.v + Rn.beta.v), W = half * (L.W + Rn.W);
    R u[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        u[k] = half * (L.u[k] + Rn.u[k]);
        b[k] *= half;
    }
    const R hbe = half * be;
    bsq *= half;
    c *= half;
    Wb0 *= half;
    vn *= half;
    un *= half;
    Bn *= half;
    const R Lam = W * W - (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]), al0 = (R)1 + gm1inv * ibln;
    const R iW = qrcp<R>(W), ibe = qrcp<R>(be), iLam = qrcp<R>(Lam);
    // U~ up to its solve for U5, times mt; F~ along m
    const R Bb0 = half * Bn * b0m, h0 = rm + hbe * bsq, h1 = hbe * Wb0 * iW;
    const R X1 = vn * Wb0 + Bb0, X2 = vn * c + Bn, bi = be * iW, cc = -bi * X2, cW = bi * iW * X1;
    const R al1 = h0 + h1, hm = h0 - h1, rW = rln * W, ru_n = rln * un;
    R R1 = half * (half * Wbsq - Wb0) - al0 * rW, T = (R)0, uru = (R)0;
    R acc = al0 * ru_n - (half * half) * Sn + Bb0;
    R UB[3], FB[3], G[3];
    const R ciW = c * iW, a1 = al1 * iW, bec = bi * c, cb = cc * ibe;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        UB[k] = W * b[k] - ciW * u[k];
        R1 -= b[k] * UB[k];
        const R Rk = a1 * u[k] - bec * b[k];
        T += u[k] * Rk;
        R ru = cW * u[k] + cc * b[k];
        if (k < NJ) ru += m[k] * hm;
        FB[k] = un * b[k] + cb * u[k];
        uru += u[k] * ru;
        acc += b[k] * FB[k];
        G[k] = mt * Rk + ru;
    }
    T -= be * R1;
    // the energy components of mt U~ + F~
    const R E = W * iLam * (ibe * (mt * T + uru) + acc), Eu = E * iW;
    out[0] = mt * rW + ru_n;
    out[4] = E;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        out[1 + k] = G[k] * ibe + Eu * u[k];
        out[5 + k] = mt * UB[k] + FB[k];
    }
}

// ---------------------------------------------------------------------------
// Per padded node: recovery (warm-started from zg_in), node values, metrics.
template <int P>
__global__ void __maxnreg__(64) k_node_mhd(ProbArg pa, double gam, const double *__restrict__ cons, const double *__restrict__ J,
                           const double *__restrict__ x, const double *__restrict__ xdot,
                           const double *__restrict__ zg_in, double *__restrict__ zg_out, double *__restrict__ q,
                           int *__restrict__ status, const double *__restrict__ inflow, int f32_logs,
                           float *__restrict__ q32)
{
    ProbDesc D;
    long long lb;
    locate(pa, D, lb);
    const Geom &g = D.g;
    long long t = lb * blockDim.x + threadIdx.x;
    if (t >= g.P) return;
    int I = (int)(t % g.px) - GH, Jn = (int)(t / g.px) - GH;
    long long src = data_src(g, I, Jn);
    double iJ = qrcp<double>(J[src]);
    double U[8], w[8], Z;
#pragma unroll
    for (int a = 0; a < 8; ++a) U[a] = cons[a * g.N + src] * iJ;
    int st = 0;
    if (inflow && ((g.bc0 == 2 && I < 0) || (g.bc1 == 2 && Jn < 0))) {
        // a ghost beyond an inflow end: the given state
        for (int a = 0; a < 8; ++a) w[a] = inflow[a];
        Z = 0.0;
    } else {
        st = cons2prim_mhd(gam, U, zg_in ? zg_in[src] : -1.0, w, Z);
    }
    bool interior = I >= 0 && I < g.nx && Jn >= 0 && Jn < g.ny;
    if (interior) {
        if (st) atomicAdd(status, 1);
        if (zg_out) zg_out[src] = Z;
    }
    const double W = qrsq<double>(1.0 - (w[1] * w[1] + w[2] * w[2] + w[3] * w[3]));
    const double beta = w[0] * qrcp<double>(w[4]);
    q[Q_RHO * g.P + t] = w[0];
    q[Q_P * g.P + t] = w[4];
    q[Q_BETA * g.P + t] = beta;
    q[Q_UX * g.P + t] = W * w[1];
    q[Q_UY * g.P + t] = W * w[2];
    q[QM_UZ * g.P + t] = W * w[3];
    q[Q_W * g.P + t] = W;
    // (f32_logs: the mixed form's scheme passes, where the logarithms enter only FP32
    // arithmetic)
    float lr32 = 0.0f, lb32 = 0.0f;
    if (f32_logs) {
        lr32 = logf(d2f_int(w[0]));
        lb32 = logf(d2f_int(beta));
    }
    const double lr = f32_logs ? f2d_int(lr32) : log(w[0]), lb_ = f32_logs ? f2d_int(lb32) : log(beta);
    q[Q_LNR * g.P + t] = lr;
    q[Q_LNB * g.P + t] = lb_;
    q[QM_B1 * g.P + t] = w[5];
    q[QM_B2 * g.P + t] = w[6];
    q[QM_B3 * g.P + t] = w[7];
    if (q32) {
        const LmV<float> r = lmv_f32(w[0], d2f_int(w[0]), f32_logs ? lr32 : d2f_int(lr));
        const LmV<float> b = lmv_f32(beta, d2f_int(beta), f32_logs ? lb32 : d2f_int(lb_));
        q32[QM32_R * g.P + t] = r.v;
        q32[QM32_RLO * g.P + t] = r.lo;
        q32[QM32_LNR * g.P + t] = r.l;
        q32[QM32_B * g.P + t] = b.v;
        q32[QM32_BLO * g.P + t] = b.lo;
        q32[QM32_LNB * g.P + t] = b.l;
        q32[QM32_W * g.P + t] = d2f_int(W);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            q32[(QM32_U0 + k) * g.P + t] = d2f_int(W * w[1 + k]);
            q32[(QM32_B0 + k) * g.P + t] = d2f_int(w[5 + k]);
        }
    }
    double dxi_x = 0.0, dxi_y = 0.0, deta_x = 0.0, deta_y = 0.0;
#pragma unroll
    for (int n = 1; n <= P; ++n) {
        const double a = 0.5 * (P == 1 ? 1.0 : (P == 2 ? (n == 1 ? 4.0 / 3.0 : -1.0 / 6.0)
                                                        : (n == 1 ? 1.5 : (n == 2 ? -0.3 : 1.0 / 30.0))));
        dxi_x += a * (mesh_at(g, x, I + n, Jn, 0, 1) - mesh_at(g, x, I - n, Jn, 0, 1));
        dxi_y += a * (mesh_at(g, x, I + n, Jn, 1, 1) - mesh_at(g, x, I - n, Jn, 1, 1));
        deta_x += a * (mesh_at(g, x, I, Jn + n, 0, 1) - mesh_at(g, x, I, Jn - n, 0, 1));
        deta_y += a * (mesh_at(g, x, I, Jn + n, 1, 1) - mesh_at(g, x, I, Jn - n, 1, 1));
    }
    double M00 = deta_y, M01 = -deta_x, M10 = -dxi_y, M11 = dxi_x;
    q[Q_M00 * g.P + t] = M00;
    q[Q_M01 * g.P + t] = M01;
    q[Q_M10 * g.P + t] = M10;
    q[Q_M11 * g.P + t] = M11;
    double xd = 0.0, yd = 0.0;
    if (xdot) { xd = mesh_at(g, xdot, I, Jn, 0, 0); yd = mesh_at(g, xdot, I, Jn, 1, 0); }
    q[Q_MT0 * g.P + t] = -(xd * M00 + yd * M01);
    q[Q_MT1 * g.P + t] = -(xd * M10 + yd * M11);
}

// entropy variables of a node from its stored values: V = (Gamma/(Gamma-1) +
// ln rho + ln beta/(Gamma-1) + beta, beta u, -beta W, beta b)
template <typename R>
__device__ __forceinline__ void node_V_mhd(const R *__restrict__ v, long long P, long long c, R c1g, R ig, R V[8])
{
    using I = NodeIx<R>;
    const R beta = v[I::BETA * P + c], W = v[I::W * P + c];
    const R u0 = v[I::U0 * P + c], u1 = v[I::U1 * P + c], u2 = v[I::U2 * P + c];
    const R B0 = v[I::B0 * P + c], B1 = v[I::B1 * P + c], B2 = v[I::B2 * P + c];
    const R b0 = u0 * B0 + u1 * B1 + u2 * B2;
    const R bW = beta * qrcp<R>(W);
    V[0] = c1g + v[I::LNR * P + c] + ig * v[I::LNB * P + c] + beta;
    V[1] = beta * u0;
    V[2] = beta * u1;
    V[3] = beta * u2;
    V[4] = -beta * W;
    V[5] = bW * (B0 + b0 * u0);
    V[6] = bW * (B1 + b0 * u1);
    V[7] = bW * (B2 + b0 * u2);
}

// Bound: FP64 the FP64 pipe (3,150 instructions per interface at p = 2, w = 5, 19 cycles of
// an SM each per warp: 1.57 ms a sweep of 512^2, all of it), FP32 instruction issue (50%, 20
// warps an SM; 128 registers take 3.63 ms for two mixed 512^2 steps, 168 3.85 and 96
// 3.84).  Measured with the pair flux along the metric vector, jumps from differences,
// the scalar form of the waves, turned pairs and the FP32 node copies: two 512^2 rotor
// steps 40.0 -> 23.2 ms, mixed 6.1 -> 3.6 ms; 64^3 blast step 32.9 -> 21.0 ms; a 160^2 p = 3
// step without dissipation 1.42 -> 0.95 ms.
// ES interface flux (eq. ESFlux_HO) between node L in [-1, n_dir - 1] and
// L + 1: the 2p-th order EC sum of two-point fluxes (eq. ECFlux_O2p, summed
// directly), the metric flux (eq. MetricsFlux_O2p), the magnetic flux B~
// (eqs. BFlux_O2p / BFlux_O2) and the WENO dissipation on scaled entropy
// variables at the interface state rho = {{rho}}^ln, u = {{u}},
// p = {{rho}}/{{beta}}, B = {{B}}.
template <typename R, int P, int WW>
__global__ void __launch_bounds__(128, sizeof(R) == 4 ? 4 : 1) k_iface_mhd(ProbArg pa, Phys ph, const double *__restrict__ q,
                                                   const R *__restrict__ qr, R *__restrict__ iflux, int dir)
{
    ProbDesc D;
    long long lb;
    locate(pa, D, lb);
    const Geom &g = D.g;
    const int nd = dir == 0 ? g.nx : g.ny, no = dir == 0 ? g.ny : g.nx;
    const long long count = (long long)(nd + 1) * no;
    const long long idx = lb * blockDim.x + threadIdx.x;
    if (idx >= count) return;
    int i, j;
    if (dir == 0) { j = (int)(idx / (nd + 1)); i = (int)(idx % (nd + 1)) - 1; }
    else { i = (int)(idx % no); j = (int)(idx / no) - 1; }
    const long long c0 = pidx(g, i, j);
    const long long sd = dir == 0 ? 1 : g.px;
    const double *Mt = q + (Q_MT0 + dir) * g.P;
    const double *Mx = q + (Q_M00 + 2 * dir) * g.P;
    const double *My = q + (Q_M01 + 2 * dir) * g.P;
    const double *B1 = q + QM_B1 * g.P, *B2 = q + QM_B2 * g.P;
    const R gm1inv = (R)(1.0 / (ph.gamma - 1.0));

    R F[8] = {(R)0, (R)0, (R)0, (R)0, (R)0, (R)0, (R)0, (R)0};
    double Ft = 0.0, Bt = 0.0;
    // (rolled in FP32, for instruction fetch, as in each_index)
#pragma unroll (sizeof(R) == 4 ? 1 : P)
    for (int n = 1; n <= P; ++n) {
        R Fs[8] = {(R)0, (R)0, (R)0, (R)0, (R)0, (R)0, (R)0, (R)0};
        double Fts = 0.0, Bts = 0.0;
#pragma unroll (sizeof(R) == 4 ? 1 : P)
        for (int s = 0; s < n; ++s) {
            const long long cl = c0 - s * sd, cr = cl + n * sd;
            NodeMT<R> l = load_node_m<R>(qr, g.P, cl), r = load_node_m<R>(qr, g.P, cr);
            R out[8];
            const double mx = Mx[cl] + Mx[cr], my = My[cl] + My[cr], mt = Mt[cl] + Mt[cr];
            const R mm[3] = {in_w<R>(0.5 * mx), in_w<R>(0.5 * my), (R)0};
            ec_pair_mhd<2, R>(l, r, gm1inv, ph.ln_thr, in_w<R>(0.5 * mt), mm, out);
#pragma unroll
            for (int a = 0; a < 8; ++a) Fs[a] += out[a];
            Fts += mt;
            Bts += mx * (B1[cl] + B1[cr]) + my * (B2[cl] + B2[cr]);
        }
        const R an = (R)ph.alpha[n - 1];
#pragma unroll
        for (int a = 0; a < 8; ++a) F[a] += an * Fs[a];
        Ft += 0.5 * ph.alpha[n - 1] * Fts;
        Bt += 0.25 * ph.alpha[n - 1] * Bts;
    }

    if constexpr (WW > 0) {
        constexpr int OFF = (WW - 1) / 2;
        const R half = (R)0.5;
        const long long c1 = c0 + sd;
        const R nvx = in_w<R>(0.5 * (Mx[c0] + Mx[c1])), nvy = in_w<R>(0.5 * (My[c0] + My[c1]));
        const R jt = in_w<R>(0.5 * (Mt[c0] + Mt[c1]));
        const R n2 = nvx * nvx + nvy * nvy, iLk = qrsq<R>(n2), Lk = n2 * iLk, nx = nvx * iLk, ny = nvy * iLk;
        // interface state, rotated
        R rho, p, ip, us[3], Bs[3];
        {
            const NodeMT<R> l = load_node_m<R>(qr, g.P, c0), r = load_node_m<R>(qr, g.P, c1);
            R irho;
            logmean2<R>(l.rho, r.rho, ph.ln_thr, rho, irho);
            const R sr = l.rho.v + r.rho.v, sb = l.beta.v + r.beta.v;
            p = sr * qrcp<R>(sb);
            ip = sb * qrcp<R>(sr);
            R um[3], Bm[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                um[k] = half * (l.u[k] + r.u[k]);
                Bm[k] = half * (l.B[k] + r.B[k]);
            }
            us[0] = nx * um[0] + ny * um[1];
            us[1] = nx * um[1] - ny * um[0];
            us[2] = um[2];
            Bs[0] = nx * Bm[0] + ny * Bm[1];
            Bs[1] = nx * Bm[1] - ny * Bm[0];
            Bs[2] = Bm[2];
        }
        const R ig = gm1inv, c1g = (R)ph.gamma * gm1inv;
        R d[8];
        es_dissipation_mhd<R, WW>(ph, rho, p, ip, us, Bs, Lk, jt, [&](int k, R TV[8]) {
            R V[8];
            node_V_mhd<R>(qr, g.P, c0 + (k - OFF) * sd, c1g, ig, V);
            TV[0] = V[0];
            TV[1] = nx * V[1] + ny * V[2];
            TV[2] = nx * V[2] - ny * V[1];
            TV[3] = V[3];
            TV[4] = V[4];
            TV[5] = nx * V[5] + ny * V[6];
            TV[6] = nx * V[6] - ny * V[5];
            TV[7] = V[7];
        }, d);
        F[0] -= d[0];
        F[1] -= nx * d[1] - ny * d[2];
        F[2] -= ny * d[1] + nx * d[2];
        F[3] -= d[3];
        F[4] -= d[4];
        F[5] -= nx * d[5] - ny * d[6];
        F[6] -= ny * d[5] + nx * d[6];
        F[7] -= d[7];
    }
    R *out = iflux + (long long)(dir * NFM) * g.P + c0;
#pragma unroll
    for (int a = 0; a < 8; ++a) out[a * g.P] = F[a];
    out[8 * g.P] = in_w<R>(Ft);
    out[9 * g.P] = in_w<R>(Bt);
}

// initial J and cons = J U(prim)
template <int P>
__global__ void k_init_state_mhd(ProbArg pa, double gam, const double *__restrict__ prim,
                                 const double *__restrict__ x, double *__restrict__ cons, double *__restrict__ J,
                                 int *status)
{
    ProbDesc D;
    long long lb;
    locate(pa, D, lb);
    const Geom &g = D.g;
    long long id = lb * blockDim.x + threadIdx.x;
    if (id >= g.N) return;
    int i = (int)(id % g.nx), j = (int)(id / g.nx);
    double dxi_x = 0.0, dxi_y = 0.0, deta_x = 0.0, deta_y = 0.0;
#pragma unroll
    for (int n = 1; n <= P; ++n) {
        const double a = 0.5 * (P == 1 ? 1.0 : (P == 2 ? (n == 1 ? 4.0 / 3.0 : -1.0 / 6.0)
                                                        : (n == 1 ? 1.5 : (n == 2 ? -0.3 : 1.0 / 30.0))));
        dxi_x += a * (mesh_at(g, x, i + n, j, 0, 1) - mesh_at(g, x, i - n, j, 0, 1));
        dxi_y += a * (mesh_at(g, x, i + n, j, 1, 1) - mesh_at(g, x, i - n, j, 1, 1));
        deta_x += a * (mesh_at(g, x, i, j + n, 0, 1) - mesh_at(g, x, i, j - n, 0, 1));
        deta_y += a * (mesh_at(g, x, i, j + n, 1, 1) - mesh_at(g, x, i, j - n, 1, 1));
    }
    double J0 = dxi_x * deta_y - deta_x * dxi_y;
    double w[8], U[8], F[8], V[8];
#pragma unroll
    for (int a = 0; a < 8; ++a) w[a] = prim[a * g.N + id];
    double v2 = w[1] * w[1] + w[2] * w[2] + w[3] * w[3];
    if (!(w[0] > 0.0) || !(w[4] > 0.0) || !(v2 < 1.0) || !(J0 > 0.0)) {
        atomicAdd(status + 1, 1);
        w[0] = 1.0; w[4] = 1.0; w[1] = w[2] = w[3] = 0.0;   // keep the arithmetic finite
    }
    mhd_UFV<double>(gam, w, U, F, V);
    J[id] = J0;
#pragma unroll
    for (int a = 0; a < 8; ++a) cons[a * g.N + id] = J0 * U[a];
}

// d/dt = -sum_k (F_k(i+1/2) - F_k(i-1/2)) - Phi'(V_i) sum_k (B~_k(i+1/2) -
// B~_k(i-1/2)) (eq. RMHDSemiU_O2p_ES), dJ/dt from the metric flux; written
// out (dcons != NULL) or combined into the SSP-RK3 stage as in k_update.
template <typename R>
__global__ void k_update_mhd(ProbArg pa, const double *__restrict__ q, const R *__restrict__ fl,
                             double *__restrict__ dcons, double *__restrict__ dJ, const double *__restrict__ cn,
                             const double *__restrict__ Jn_, const double *__restrict__ xn,
                             const double *__restrict__ cs, const double *__restrict__ Js,
                             const double *__restrict__ xs, const double *__restrict__ xdot, double A, double B,
                             const double *__restrict__ dt_dev, double *__restrict__ co, double *__restrict__ Jo,
                             double *__restrict__ xo)
{
    ProbDesc D;
    long long lb;
    int b = locate(pa, D, lb);
    const Geom &g = D.g;
    long long id = lb * blockDim.x + threadIdx.x;
    if (id >= g.N) return;
    int i = (int)(id % g.nx), j = (int)(id / g.nx);
    long long c = pidx(g, i, j);
    const R *f0 = fl, *f1 = fl + NFM * g.P;
    double L[10];
#pragma unroll
    for (int a = 0; a < 10; ++a) {
        double d0 = to_f64(f0[a * g.P + c]) - to_f64(f0[a * g.P + c - 1]);
        double d1 = to_f64(f1[a * g.P + c]) - to_f64(f1[a * g.P + c - g.px]);
        L[a] = -(d0 + d1);
    }
    // Powell source: L[9] = -div B~ here
    const double iW = qrcp<double>(q[Q_W * g.P + c]);
    double w[8];
    w[1] = q[Q_UX * g.P + c] * iW;
    w[2] = q[Q_UY * g.P + c] * iW;
    w[3] = q[QM_UZ * g.P + c] * iW;
    w[5] = q[QM_B1 * g.P + c];
    w[6] = q[QM_B2 * g.P + c];
    w[7] = q[QM_B3 * g.P + c];
    double Pp[8];
    mhd_phiprime(w, Pp);
#pragma unroll
    for (int a = 1; a < 8; ++a) L[a] += Pp[a] * L[9];   // (Phi'_1 = 0)
    if (dcons) {
#pragma unroll
        for (int a = 0; a < 8; ++a) dcons[a * g.N + id] = L[a];
        dJ[id] = L[8];
        return;
    }
    double dt = dt_dev[b];
#pragma unroll
    for (int a = 0; a < 8; ++a) co[a * g.N + id] = A * cn[a * g.N + id] + B * (cs[a * g.N + id] + dt * L[a]);
    Jo[id] = A * Jn_[id] + B * (Js[id] + dt * L[8]);
    xo[id] = A * xn[id] + B * (xs[id] + dt * xdot[id]);
    xo[g.N + id] = A * xn[g.N + id] + B * (xs[g.N + id] + dt * xdot[g.N + id]);
}


#if defined(__CUDACC__)
template <typename R, int P>
static void launch_iface_mhd_p(const LaunchDom &L, const Phys &ph, const double *q, const R *qr, R *iflux, int dir,
                               cudaStream_t st)
{
    switch (ph.w) {
    case 0: k_iface_mhd<R, P, 0><<<L.nblk, L.bs, 0, st>>>(L.pa, ph, q, qr, iflux, dir); break;
    case 3: k_iface_mhd<R, P, 3><<<L.nblk, L.bs, 0, st>>>(L.pa, ph, q, qr, iflux, dir); break;
    default: k_iface_mhd<R, P, 5><<<L.nblk, L.bs, 0, st>>>(L.pa, ph, q, qr, iflux, dir); break;
    }
}

// interface fluxes of one sweep direction in the working precision R
template <typename R>
static void launch_iface_mhd_t(const LaunchDom &L, const Phys &ph, const double *q, const R *qr, void *iflux, int dir,
                               cudaStream_t st)
{
    R *fl = (R *)iflux;
    switch (ph.p) {
    case 1: launch_iface_mhd_p<R, 1>(L, ph, q, qr, fl, dir, st); break;
    case 2: launch_iface_mhd_p<R, 2>(L, ph, q, qr, fl, dir, st); break;
    default: launch_iface_mhd_p<R, 3>(L, ph, q, qr, fl, dir, st); break;
    }
}

template <typename R>
static void launch_update_mhd_t(const LaunchDom &L, const double *q, const void *fl, double *dcons, double *dJ,
                                const double *cn, const double *Jn, const double *xn, const double *cs,
                                const double *Js, const double *xs, const double *xdot, double A, double B,
                                const double *dt_dev, double *co, double *Jo, double *xo, cudaStream_t st)
{
    k_update_mhd<R><<<L.nblk, L.bs, 0, st>>>(L.pa, q, (const R *)fl, dcons, dJ, cn, Jn, xn, cs, Js, xs, xdot, A, B,
                                             dt_dev, co, Jo, xo);
}
#endif

}  // namespace esmm

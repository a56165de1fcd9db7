// esmm_mhd_vjp.cuh -- reverse sweeps of the RMHD flux arithmetic, shared by the
// 2D and the 3D adjoint (esmm_mhd_adjoint.cu, esmm_3d_adjoint.cu): the two-point
// flux, the WENO jump, and the ES dissipation through the eigen-system.
//
// The eigen-system's adjoint is first-order perturbation theory on the eight
// waves: with the symmetric forms G = U_w^T V_w and K = V_w^T F~_w (columns: the
// primitive directions) and the waves a_m (a^T G a = 1, speeds lambda_m),
//   a_m' = sum_n c_nm a_n,   c_nm = a_n^T (K' - lambda_m G') a_m / (lambda_m - lambda_n),
//   c_mm = -1/2 a_m^T G' a_m,   lambda_m' = a_m^T (K' - lambda_m G') a_m,
// and for n the entropy or the divergence wave (fixed directions of the state) the
// coefficient that keeps a_n^T G a_m = 0.  Every term is linear in U_w', V_w' and
// F~_w', so the objective's gradient is, per wave, the derivative along a_m of the
// gradient of alpha_U.U + alpha_V.V + alpha_F.F: one reverse sweep of (U, F, V) on
// dual numbers.  That replaces one whole eigen-system with tangents (Gram matrix on
// hyper-dual images, Jacobi) per state direction, eight per interface.
// Bound: the FP64 pipe and the ~5 KB frame of the 8 x 8 arrays in local memory.
// Measured (GB300): the vector-Jacobian product of 32^3 nodes 57 -> 2.9 ms, of a 48^3
// blast, whose speeds cluster everywhere, 158 -> 13.9 ms; two recorded 96^2 steps and
// their gradient 147 -> 13.0 ms.
#pragma once

#include "esmm_mhd.cuh"
#include "esmm_vjp.cuh"

namespace esmm {

enum { A_RHO = 0, A_BETA, A_LNR, A_LNB, A_W, A_U0, A_U1, A_U2, A_B0, A_B1, A_B2, NQN };

// Adjoint of ec_pair_mhd: lp the adjoint of its eight components, lbs that of the
// pair's magnetic flux 1/2 m.(B_l + B_r); gL, gR receive the adjoints of the node
// quantities.  The flux is linear in the metric vector m, so its spatial part is
// taken once, contracted with m.
__device__ __forceinline__ void mhd_pair_vjp(const NodeM &L, const NodeM &Rn, double gm1inv, double thr, double mt,
                                             const double m[3], const double lp[8], double lbs, double gL[NQN],
                                             double gR[NQN])
{
    double rln, irln, bln, ibln;
    logmean<double, double>(L.rho.v, Rn.rho.v, L.rho.l, Rn.rho.l, thr, rln, irln);
    logmean<double, double>(L.beta.v, Rn.beta.v, L.beta.l, Rn.beta.l, thr, bln, ibln);
    double bX[2][3], b0X[2], iWX[2], bbX[2], unX[2], BnX[2];
    const NodeM *N[2] = {&L, &Rn};
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        const NodeM &n = *N[x];
        b0X[x] = n.u[0] * n.B[0] + n.u[1] * n.B[1] + n.u[2] * n.B[2];
        iWX[x] = __drcp_rn(n.W);
        for (int k = 0; k < 3; ++k) bX[x][k] = (n.B[k] + b0X[x] * n.u[k]) * iWX[x];
        bbX[x] = bX[x][0] * bX[x][0] + bX[x][1] * bX[x][1] + bX[x][2] * bX[x][2];
        unX[x] = m[0] * n.u[0] + m[1] * n.u[1] + m[2] * n.u[2];
        BnX[x] = m[0] * n.B[0] + m[1] * n.B[1] + m[2] * n.B[2];
    }
    const double rm = 0.5 * (L.rho.v + Rn.rho.v), be = 0.5 * (L.beta.v + Rn.beta.v), W = 0.5 * (L.W + Rn.W);
    double u[3], b[3];
    for (int k = 0; k < 3; ++k) {
        u[k] = 0.5 * (L.u[k] + Rn.u[k]);
        b[k] = 0.5 * (bX[0][k] + bX[1][k]);
    }
    const double bsq = 0.5 * (bbX[0] + bbX[1]), Wbsq = 0.5 * (L.W * bbX[0] + Rn.W * bbX[1]);
    const double c = 0.5 * (L.W * b0X[0] + Rn.W * b0X[1]), b0m = 0.5 * (b0X[0] + b0X[1]);
    const double Wb0 = 0.5 * (L.W * b0X[0] * b0X[0] + Rn.W * b0X[1] * b0X[1]);
    const double Sn = 0.5 * (unX[0] * bbX[0] + unX[1] * bbX[1]);
    const double S0n = 0.5 * (unX[0] * b0X[0] * b0X[0] + unX[1] * b0X[1] * b0X[1]);
    const double vn = 0.5 * (unX[0] * iWX[0] + unX[1] * iWX[1]), Bn = 0.5 * (BnX[0] + BnX[1]), un = 0.5 * (unX[0] + unX[1]);
    const double usq = u[0] * u[0] + u[1] * u[1] + u[2] * u[2], Lam = W * W - usq, al0 = 1.0 + gm1inv * ibln;
    const double iW = __drcp_rn(W), ibe = __drcp_rn(be), iLam = __drcp_rn(Lam);
    // forward, temporal part
    const double al1 = rm + 0.5 * be * bsq + 0.5 * be * Wb0 * iW, U1 = rln * W;
    double UB[3], Rk[3], R1 = -al0 * U1 - 0.5 * Wb0 + 0.5 * Wbsq, T = 0.0;
    for (int k = 0; k < 3; ++k) {
        UB[k] = W * b[k] - c * u[k] * iW;
        R1 -= b[k] * UB[k];
        Rk[k] = (al1 * u[k] - be * c * b[k]) * iW;
        T += u[k] * Rk[k];
    }
    T -= be * R1;
    const double U5 = T * W * ibe * iLam;
    // forward, spatial part along m
    const double X1 = vn * Wb0 + Bn * b0m, X2 = vn * c + Bn, cc = -be * iW * X2, cW = be * iW * X1;
    const double h = rm + 0.5 * be * bsq - 0.5 * be * Wb0 * iW, rbeta = 0.5 * Sn - 0.5 * S0n - Bn * b0m;
    double ru[3], FB[3], acc = 0.0, uru = 0.0;
    for (int k = 0; k < 3; ++k) {
        ru[k] = m[k] * h + cW * iW * u[k] + cc * b[k];
        FB[k] = un * b[k] + cc * ibe * u[k];
        uru += u[k] * ru[k];
        acc += b[k] * FB[k];
    }
    acc += al0 * rln * un - rbeta + ibe * uru;
    const double F4 = W * iLam * acc;
    // reverse, spatial part
    double gu[3], gb[3], gru[3], gFB[3], gW = 0.0, giW, gib, giL, ga0, grln, gun, gcc = 0.0, gbe, gc, gWb0, gbsq, grm;
    double t1 = 0.0, t2 = 0.0, t3 = 0.0;
    for (int k = 0; k < 3; ++k) {
        t1 += lp[1 + k] * u[k];
        t2 += lp[1 + k] * ru[k];
    }
    const double gF4 = lp[4] + t1 * iW;
    giW = F4 * t1;
    const double gac = gF4 * W * iLam;
    gW += gF4 * iLam * acc;
    giL = gF4 * W * acc;
    gib = t2 + gac * uru;
    const double F0 = rln * un, gF0 = lp[0] + gac * al0;
    ga0 = gac * F0;
    for (int k = 0; k < 3; ++k) {
        gu[k] = lp[1 + k] * F4 * iW + gac * ibe * ru[k];
        gru[k] = (lp[1 + k] + gac * u[k]) * ibe;
        gb[k] = gac * FB[k];
        gFB[k] = lp[5 + k] + gac * b[k];
        t3 += gFB[k] * u[k];
    }
    gun = gF0 * rln;
    grln = gF0 * un;
    double gh = 0.0, t4 = 0.0;
    for (int k = 0; k < 3; ++k) {
        gun += gFB[k] * b[k];
        gb[k] += gFB[k] * un + gru[k] * cc;
        gu[k] += gFB[k] * cc * ibe + gru[k] * cW * iW;
        gh += gru[k] * m[k];
        t4 += gru[k] * u[k];
        gcc += gru[k] * b[k];
    }
    gcc += t3 * ibe;
    gib += t3 * cc;
    const double gcW = t4 * iW;
    giW += t4 * cW;
    grm = gh;
    gbe = gh * (0.5 * bsq - 0.5 * Wb0 * iW) + gcW * iW * X1 - gcc * iW * X2;
    gbsq = 0.5 * be * gh;
    gWb0 = -0.5 * be * iW * gh + gcW * be * iW * vn;
    giW += -0.5 * be * Wb0 * gh + gcW * be * X1 - gcc * be * X2;
    const double gvn = gcW * be * iW * Wb0 - gcc * be * iW * c;
    gc = -gcc * be * iW * vn;
    const double gBn = gcW * be * iW * b0m - gcc * be * iW + gac * b0m + lbs;
    const double gb0m = gcW * be * iW * Bn + gac * Bn;
    const double gSn = -0.5 * gac, gS0n = 0.5 * gac;
    // reverse, temporal part
    double gU1 = mt * lp[0], gRk[3], gUB[3], q1 = 0.0, q2 = 0.0;
    for (int k = 0; k < 3; ++k) {
        q1 += lp[1 + k] * u[k];
        q2 += lp[1 + k] * Rk[k];
    }
    const double gU5 = mt * (lp[4] + q1 * iW);
    giW += mt * U5 * q1;
    gib += mt * q2;
    const double gT = gU5 * W * ibe * iLam;
    gW += gU5 * T * ibe * iLam;
    gib += gU5 * T * W * iLam;
    giL += gU5 * T * W * ibe;
    const double gR1 = -gT * be;
    gbe -= gT * R1;
    ga0 -= gR1 * U1;
    gU1 -= gR1 * al0;
    gWb0 -= 0.5 * gR1;
    const double gWbsq = 0.5 * gR1;
    double s1 = 0.0, s2 = 0.0, s3 = 0.0, s4 = 0.0;
    for (int k = 0; k < 3; ++k) {
        gu[k] += mt * lp[1 + k] * U5 * iW + gT * Rk[k];
        gRk[k] = mt * lp[1 + k] * ibe + gT * u[k];
        gUB[k] = mt * lp[5 + k] - gR1 * b[k];
        gb[k] -= gR1 * UB[k];
        s1 += gRk[k] * u[k];
        s2 += gRk[k] * b[k];
        s3 += gUB[k] * b[k];
        s4 += gUB[k] * u[k];
    }
    const double ga1 = s1 * iW;
    gbe -= s2 * c * iW;
    gc -= s2 * be * iW + iW * s4;
    giW += s1 * al1 - s2 * be * c - c * s4;
    gW += s3 + gU1 * rln;
    for (int k = 0; k < 3; ++k) {
        gu[k] += gRk[k] * al1 * iW - gUB[k] * c * iW;
        gb[k] += gUB[k] * W - gRk[k] * be * c * iW;
    }
    grm += ga1;
    gbe += ga1 * (0.5 * bsq + 0.5 * Wb0 * iW);
    gbsq += 0.5 * be * ga1;
    gWb0 += 0.5 * be * iW * ga1;
    giW += 0.5 * be * Wb0 * ga1;
    grln += gU1 * W;
    const double gLam = -giL * iLam * iLam;
    gW += 2.0 * W * gLam - giW * iW * iW;
    for (int k = 0; k < 3; ++k) gu[k] -= 2.0 * u[k] * gLam;
    gbe -= gib * ibe * ibe;
    // to the nodes
    double *go[2] = {gL, gR};
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        const NodeM &n = *N[x];
        double *g = go[x];
        double gbk[3], gWx = 0.5 * gW + 0.5 * bbX[x] * gWbsq + 0.5 * b0X[x] * gc + 0.5 * b0X[x] * b0X[x] * gWb0;
        double gb0 = 0.5 * n.W * gc + n.W * b0X[x] * gWb0 + 0.5 * gb0m + unX[x] * b0X[x] * gS0n;
        const double cb = gbsq + n.W * gWbsq + unX[x] * gSn;
        const double gun_x = 0.5 * (bbX[x] * gSn + b0X[x] * b0X[x] * gS0n + iWX[x] * gvn + gun);
        double giWx = 0.5 * unX[x] * gvn;
        for (int k = 0; k < 3; ++k) {
            gbk[k] = 0.5 * gb[k] + bX[x][k] * cb;
            gb0 += iWX[x] * gbk[k] * n.u[k];
            giWx += gbk[k] * (n.B[k] + b0X[x] * n.u[k]);
        }
        for (int k = 0; k < 3; ++k) {
            g[A_U0 + k] = 0.5 * gu[k] + m[k] * gun_x + gbk[k] * b0X[x] * iWX[x] + gb0 * n.B[k];
            g[A_B0 + k] = 0.5 * m[k] * gBn + gbk[k] * iWX[x] + gb0 * n.u[k];
        }
        g[A_W] = gWx - giWx * iWX[x] * iWX[x];
        g[A_RHO] = 0.5 * grm;
        g[A_BETA] = 0.5 * gbe;
        g[A_LNR] = 0.0;
        g[A_LNB] = 0.0;
    }
    logmean_vjp(L.rho.v, Rn.rho.v, L.rho.l, Rn.rho.l, thr, grln, gL[A_RHO], gR[A_RHO], gL[A_LNR], gR[A_LNR]);
    logmean_vjp(L.beta.v, Rn.beta.v, L.beta.l, Rn.beta.l, thr, -ga0 * gm1inv * ibln * ibln, gL[A_BETA], gR[A_BETA], gL[A_LNB],
                gR[A_LNB]);
}

// gradient of aU.U + aF.F_1 + aV.V (mhd_UFV) with respect to the primitives
template <typename T>
__device__ __forceinline__ void mhd_UFV_grad(double gam, const T w[8], const double aU[8], const double aF[8],
                                             const double aV[8], T g[8])
{
    const double gm1i = 1.0 / (gam - 1.0), gg = gam * gm1i;
    const T rho = w[0], p = w[4];
    const T v[3] = {w[1], w[2], w[3]}, B[3] = {w[5], w[6], w[7]};
    const T iW2 = 1.0 - (v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
    const T W = rsq<T>(iW2), W2 = W * W;
    const T vB = v[0] * B[0] + v[1] * B[1] + v[2] * B[2], B2 = B[0] * B[0] + B[1] * B[1] + B[2] * B[2];
    const T rh = rho + gg * p, Q = rh * W2 + B2;
    const T ip = rcp<T>(p), beta = rho * ip, ir = rcp<T>(rho);
    T Um[3], gv[3], gB[3];
    for (int i = 0; i < 3; ++i) Um[i] = Q * v[i] - vB * B[i];
    // sums over the vector adjoints
    T eF = aF[1] * B[0] + aF[2] * B[1] + aF[3] * B[2], fF = aF[1] * v[0] + aF[2] * v[1] + aF[3] * v[2];
    T bF = aF[5] * B[0] + aF[6] * B[1] + aF[7] * B[2], vF = aF[5] * v[0] + aF[6] * v[1] + aF[7] * v[2];
    const T gU0 = aU[0] + aF[0] * v[0];
    T gUm[3];
    for (int i = 0; i < 3; ++i) gUm[i] = aU[1 + i] + aF[1 + i] * v[0] + (i == 0 ? aF[4] : 0.0);
    T gQ = gUm[0] * v[0] + gUm[1] * v[1] + gUm[2] * v[2];
    T gvB = -(gUm[0] * B[0] + gUm[1] * B[1] + gUm[2] * B[2]) - B[0] * fF;
    T giW2 = -(B[0] * eF);
    const double gpt = aF[1] - aU[4];
    const T bW = beta * iW2 * W;
    const T eB = aV[5] * B[0] + aV[6] * B[1] + aV[7] * B[2], ev = aV[5] * v[0] + aV[6] * v[1] + aV[7] * v[2];
    const T tV = aV[1] * v[0] + aV[2] * v[1] + aV[3] * v[2] - aV[4];
    const T gbW = eB + W2 * vB * ev;
    T gW2 = aU[4] * rh + gQ * rh + bW * vB * ev;
    T grh = (aU[4] + gQ) * W2;
    T gB2 = gQ + aU[4] + 0.5 * gpt * iW2;
    giW2 += 0.5 * gpt * B2;
    gvB += gpt * vB + bW * W2 * ev;
    T gbeta = aV[0] + W * tV + gbW * iW2 * W;
    giW2 += gbW * beta * W;
    T gW = gU0 * rho + beta * tV + gbW * beta * iW2 + 2.0 * (W * gW2);
    giW2 += -0.5 * (W * W2 * gW);
    const T bWW = beta * W, c5 = bW * W2 * vB;
    for (int i = 0; i < 3; ++i) {
        gv[i] = gUm[i] * Q - aF[1 + i] * (B[0] * vB) - aF[5 + i] * B[0] + aV[1 + i] * bWW + aV[5 + i] * c5 -
                2.0 * (v[i] * giW2) + gvB * B[i];
        gB[i] = aU[5 + i] - gUm[i] * vB - aF[1 + i] * (B[0] * iW2) + aF[5 + i] * v[0] + aV[5 + i] * bW + gvB * v[i] +
                2.0 * (B[i] * gB2);
    }
    gv[0] += aF[0] * (rho * W) + aF[1] * Um[0] + aF[2] * Um[1] + aF[3] * Um[2] + bF;
    gB[0] -= eF * iW2 + fF * vB + vF;
    g[0] = gU0 * W + (aV[0] * gam * gm1i) * ir + gbeta * ip + grh;
    g[4] = gpt - (aV[0] * gm1i) * ip - gbeta * beta * ip + gg * grh;
    for (int i = 0; i < 3; ++i) {
        g[1 + i] = gv[i];
        g[5 + i] = gB[i];
    }
}

// Clustered speeds: the waves of each cluster orthonormalized (R, X and A, rows 2 + m),
// the orthogonal matrix Th with canonical wave t = sum_i Th[i][t] wave i (mhd_turn_clusters),
// and what the canonical basis's derivative needs: with G_y = L L^T the Gram matrix of
// the y_a and S the waves' coefficients in them, E = L^T S (E[i][m] = <q_i, a_m>, q_i the
// Gram-Schmidt of the y_a; E of the waves, Ec of the canonical ones), rows 4 and 5 of L,
// and the index ii[t] of the unit vector that gave a cluster's member t.  A cluster's
// canonical basis is the one with Ec[ii[j]][t] = 0 for members j < t, which fixes the
// rotation within the cluster.
struct MhdClusters {
    double E[6][6], Ec[6][6], Th[6][6], L4[6], L5[6];
    int ii[6], from[6], to[6];   // cluster [from, to) of wave m
};
static __device__ __noinline__ void mhd_clusters(double gam, const double w[8], const double lam[8], double S[6][6],
                                                 double R[8][8], double X[8][8], double A[8][8], MhdClusters &c)
{
    double Pp[8];
    mhd_phiprime(w, Pp);
    const double v1 = w[1];
    const double a_rho[8] = {1, 0, 0, 0, 0, 0, 0, 0}, a_div[8] = {0, 0, 0, 0, 0, 1.0 - v1 * v1, -v1 * w[2], -v1 * w[3]};
    double Ur[8], Vr[8], Ud[8], Vd[8], Fx[8];
    mhd_images(gam, w, a_rho, Pp, Ur, Vr, Fx);
    mhd_images(gam, w, a_div, Pp, Ud, Vd, Fx);
    const double in_rho = rcp<double>(dot8(Ur, Vr)), in_div = rcp<double>(dot8(Ud, Vd));
    double Uy[6][8], Vy[6][8], Gm[6][6], idg[6], cr[6], cd[6];
#pragma unroll 1
    for (int a = 0; a < 6; ++a) {
        const int comp = a < 4 ? 1 + a : 2 + a;   // v_1, v_2, v_3, p, B_2, B_3
        double e[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        e[comp] = 1.0;
        double Ue[8], Ve[8];
        mhd_images(gam, w, e, Pp, Ue, Ve, Fx);
        cr[a] = dot8(Ue, Vr) * in_rho;
        cd[a] = dot8(Ue, Vd) * in_div;
        for (int r = 0; r < 8; ++r) {
            Uy[a][r] = Ue[r] - cr[a] * Ur[r] - cd[a] * Ud[r];
            Vy[a][r] = Ve[r] - cr[a] * Vr[r] - cd[a] * Vd[r];
        }
    }
    for (int a = 0; a < 6; ++a)
        for (int b = 0; b <= a; ++b) Gm[a][b] = 0.5 * (dot8(Uy[a], Vy[b]) + dot8(Uy[b], Vy[a]));
    for (int j = 0; j < 6; ++j) {
        double d = Gm[j][j];
        for (int k = 0; k < j; ++k) d -= Gm[j][k] * Gm[j][k];
        idg[j] = rsqrt(d);
        Gm[j][j] = d * idg[j];
        for (int i = j + 1; i < 6; ++i) {
            double s = Gm[i][j];
            for (int k = 0; k < j; ++k) s -= Gm[i][k] * Gm[j][k];
            Gm[i][j] = s * idg[j];
        }
    }
    for (int m = 0; m < 6; ++m)
        for (int i = 0; i < 6; ++i) {
            double acc = 0.0;
            for (int j = i; j < 6; ++j) acc += Gm[j][i] * S[j][m];
            c.E[i][m] = c.Ec[i][m] = acc;
            c.Th[i][m] = i == m ? 1.0 : 0.0;
        }
    for (int i = 0; i < 6; ++i) {
        c.L4[i] = i <= 4 ? Gm[4][i] : 0.0;
        c.L5[i] = Gm[5][i];
    }
    int start = 0;
    while (start < 6) {
        int end = start + 1;
        while (end < 6 && mhd_close<double>(lam[1 + end], lam[2 + end])) ++end;
        const int k = end - start;
        for (int m = start; m < end; ++m) {
            c.from[m] = start;
            c.to[m] = end;
            c.ii[m] = 0;
        }
        if (k > 1) {
            for (int q = start; q < end; ++q) {
                for (int pass = 0; pass < 2; ++pass)
                    for (int b = start; b < q; ++b) {
                        double pr = 0.0;
                        for (int i = 0; i < 6; ++i) pr += c.E[i][b] * c.E[i][q];
                        for (int i = 0; i < 6; ++i) c.E[i][q] -= pr * c.E[i][b];
                    }
                double n2 = 0.0;
                for (int i = 0; i < 6; ++i) n2 += c.E[i][q] * c.E[i][q];
                const double inr = rsqrt(n2);
                for (int i = 0; i < 6; ++i) c.E[i][q] *= inr;
                // the wave from its coefficients L^-T E
                double s[6], sr = 0.0, sdv = 0.0;
                double *r8 = R[2 + q], *x8 = X[2 + q], *a8 = A[2 + q];
                for (int i = 5; i >= 0; --i) {
                    double acc = c.E[i][q];
                    for (int j = i + 1; j < 6; ++j) acc -= Gm[j][i] * s[j];
                    s[i] = acc * idg[i];
                }
                for (int r = 0; r < 8; ++r) r8[r] = x8[r] = 0.0;
                for (int a = 0; a < 6; ++a) {
                    for (int r = 0; r < 8; ++r) {
                        r8[r] += s[a] * Uy[a][r];
                        x8[r] += s[a] * Vy[a][r];
                    }
                    sr += s[a] * cr[a];
                    sdv += s[a] * cd[a];
                }
                a8[0] = -sr;
                for (int a = 0; a < 4; ++a) a8[1 + a] = s[a];
                a8[5] = -sdv * a_div[5];
                a8[6] = s[4] - sdv * a_div[6];
                a8[7] = s[5] - sdv * a_div[7];
            }
            double z[6][6];
            for (int i = 0; i < 6; ++i)
                for (int q = 0; q < k; ++q) z[i][q] = c.E[i][start + q];
            int nt = 0;
            for (int i = 0; i < 6 && nt < k; ++i) {
                double n2 = 0.0;
                for (int q = 0; q < k; ++q) n2 += z[i][q] * z[i][q];
                if (!(n2 >= 0.125)) continue;
                const double inr = rsqrt(n2);
                for (int q = 0; q < k; ++q) c.Th[start + q][start + nt] = z[i][q] * inr;
                for (int i2 = i + 1; i2 < 6; ++i2) {
                    double pr = 0.0;
                    for (int q = 0; q < k; ++q) pr += z[i2][q] * c.Th[start + q][start + nt];
                    for (int q = 0; q < k; ++q) z[i2][q] -= pr * c.Th[start + q][start + nt];
                }
                c.ii[start + nt] = i;
                ++nt;
            }
            for (int t = start; t < end; ++t)
                for (int i = 0; i < 6; ++i) {
                    double acc = 0.0;
                    for (int q = start; q < end; ++q) acc += c.E[i][q] * c.Th[q][t];
                    c.Ec[i][t] = acc;
                }
        }
        start = end;
    }
}

// rows 2 + m of M (one per wave) to the canonical waves (fwd) or back
static __device__ __noinline__ void mhd_turn(const MhdClusters &c, double M[8][8], bool fwd)
{
#pragma unroll 1
    for (int b = 0; b < 8; ++b) {
        double o[6];
        for (int t = 0; t < 6; ++t) {
            double acc = 0.0;
            for (int q = c.from[t]; q < c.to[t]; ++q) acc += (fwd ? c.Th[q][t] : c.Th[t][q]) * M[2 + q][b];
            o[t] = acc;
        }
        for (int t = 0; t < 6; ++t) M[2 + t][b] = o[t];
    }
}

// mhd_diss_vjp by the Gram form and its tangent along each direction of the state, for what
// the closed form leaves to it (as in mhd_scaled_waves).
template <int WW>
static __device__ __noinline__ void mhd_diss_vjp_gram(const Phys &ph, const double wrot[8], double Lk, double jt,
                                                      const double lrot[8], const double TV[][8], double gTV[][8],
                                                      double gw[8], double Rz[8], double &hl)
{
    constexpr int NS = WW + 1, OFF = (WW - 1) / 2;
    double lam[8], R[8][8];   // (a column per wave)
    eigen_mhd_gram<double>(ph.gamma, wrot, lam, R, true);
    double lhat = 0.0;
    int msel = 0;
    for (int m = 0; m < 8; ++m) {
        const double v = fabs(jt + Lk * lam[m]);
        if (v > lhat) { lhat = v; msel = m; }
    }
    const double sg = (jt + Lk * lam[msel]) >= 0.0 ? 1.0 : -1.0;
    hl = 0.5 * lhat;
    for (int k = 0; k < NS; ++k)
        for (int b = 0; b < 8; ++b) gTV[k][b] = 0.0;
    for (int b = 0; b < 8; ++b) Rz[b] = 0.0;
    double Rb[8][8], zeta = 0.0;
#pragma unroll 1
    for (int m = 0; m < 8; ++m) {
        double Vt[NS], gVt[NS], scale = 0.0, qm = 0.0;
        for (int k = 0; k < NS; ++k) {
            Vt[k] = 0.0;
            for (int a = 0; a < 8; ++a) {
                const double t = R[a][m] * TV[k][a];
                Vt[k] += t;
                if (k == OFF || k == OFF + 1) scale += fabs(t);
            }
        }
        for (int b = 0; b < 8; ++b) qm += R[b][m] * lrot[b];
        double vminus, vplus;
        if constexpr (WW == 5) weno5_lr<double>(Vt[0], Vt[1], Vt[2], Vt[3], Vt[4], Vt[5], ph.eps, vminus, vplus);
        else weno3_lr<double>(Vt[0], Vt[1], Vt[2], Vt[3], ph.eps, vminus, vplus);
        const double jw = vplus - vminus, jump = Vt[OFF + 1] - Vt[OFF];
        const int sj = fabs(jump) <= ph.sign_tol * scale ? 0 : sgn_d(jump);
        const bool y = sgn_d(jw) == sj;
        const double z = y ? jw : 0.0;
        zeta += qm * z;
        for (int b = 0; b < 8; ++b) {
            Rz[b] += R[b][m] * z;
            Rb[b][m] = -hl * lrot[b] * z;
        }
        if (!y) continue;
        weno_jump_vjp<WW>(Vt, ph.eps, -hl * qm, gVt);
        for (int k = 0; k < NS; ++k)
            for (int b = 0; b < 8; ++b) {
                gTV[k][b] += R[b][m] * gVt[k];
                Rb[b][m] += gVt[k] * TV[k][b];
            }
    }
#pragma unroll 1
    for (int a = 0; a < 8; ++a) {
        dual wd[8], ld[8], Rd[8][8];
        for (int k = 0; k < 8; ++k) wd[k] = dual(wrot[k], k == a ? 1.0 : 0.0);
        eigen_mhd_gram<dual>(ph.gamma, wd, ld, Rd, true);
        double acc = -0.5 * sg * Lk * ld[msel].d * zeta;
        for (int b = 0; b < 8; ++b)
            for (int m = 0; m < 8; ++m) acc += Rb[b][m] * Rd[b][m].d;
        gw[a] = acc;
    }
}

// Reverse sweep of the ES dissipation at one interface (rotated frame):
// lrot = T lambda_F, TV the stencil's rotated entropy variables, wrot the rotated
// interface state.  gTV: adjoint of TV; gw: adjoint of wrot; Rz = R z and hl =
// lambda^/2 (for the frame's own derivative in 3D).
//
// Within a cluster of close speeds the coefficients c_nt are -1/2 a_n^T G' a_t + O_nt
// with O antisymmetric, and the conditions E[ii[j]][t] = 0 (j < t) on the canonical basis
// determine O member by member: with E' = Lam^T E + E c + a_t[B_1] L^T (h_2', h_3'), Lam the
// lower half of L^-1 G_y' L^-T and h_k = v_1 v_k/(1 - v_1^2) (from the divergence wave's
// direction), sum_{s <= j} E[ii[j]][s] O_st equals minus the rest, a triangular system
// whose adjoint adds to the coefficients of G', K' and of the divergence direction.
// The speed lambda^ keeps its own resolved wave.  False where the closed form leaves the
// interface to the Gram form.
template <int WW>
__device__ __noinline__ bool mhd_diss_vjp_waves(const Phys &ph, const double wrot[8], double Lk, double jt,
                                          const double lrot[8], const double TV[][8], double gTV[][8], double gw[8],
                                          double Rz[8], double &hl)
{
    constexpr int NS = WW + 1, OFF = (WW - 1) / 2;
    const double gam = ph.gamma, gm1i = 1.0 / (gam - 1.0), gg = gam * gm1i;
    MhdBase<double> s;
    mhd_base<double>(gam, gg, wrot, s);
    if (!mhd_in_range<double>(s)) return false;
    MhdSix<double> six;
    double lam[8];
    lam[0] = lam[1] = s.v1;
    mhd_six<double>(s, six, lam + 2);
    bool cluster = false;
    for (int m = 0; m < 5; ++m) cluster = cluster || mhd_close<double>(lam[2 + m], lam[3 + m]);
    // the waves: R (dU), X (dV), A (dw), one row per wave
    double R[8][8], X[8][8], A[8][8], S[6][6];
    const double ir = __drcp_rn(s.rho);
    double sd;
    {
        const double sr = rsqrt(gg * s.W * ir);
        for (int k = 0; k < 8; ++k) A[0][k] = A[1][k] = R[0][k] = X[0][k] = 0.0;
        A[0][0] = sr;
        R[0][0] = s.W * sr;
        for (int k = 0; k < 3; ++k) R[0][1 + k] = s.W * s.u[1 + k] * sr;
        R[0][4] = s.W * s.W * sr;
        const double db = s.ip * sr;
        X[0][0] = gg * ir * sr + db;
        for (int k = 0; k < 3; ++k) X[0][1 + k] = db * s.u[1 + k];
        X[0][4] = -db * s.W;
        for (int k = 0; k < 3; ++k) X[0][5 + k] = db * s.b[1 + k];
        MhdWave<double> q;
        const double dB[3] = {1.0 - s.v1 * s.v1, -s.v1 * wrot[2], -s.v1 * wrot[3]};
        q.rho = q.p = 0.0;
        q.b[0] = s.v1 * s.iW;
        q.u[0] = 0.0;
        for (int k = 0; k < 3; ++k) {
            q.u[1 + k] = 0.0;
            q.b[1 + k] = (dB[k] + q.b[0] * s.u[1 + k]) * s.iW;
        }
        sd = rsqrt(s.beta * s.W * mdot<double>(q.b, q.b));
        for (int k = 0; k < 4; ++k) q.b[k] *= sd;
        mhd_wave_dU<double>(s, gg, q, R[1]);
        for (int k = 0; k < 5; ++k) X[1][k] = 0.0;
        for (int k = 0; k < 3; ++k) {
            A[1][5 + k] = dB[k] * sd;
            X[1][5 + k] = s.beta * q.b[1 + k];
        }
    }
#pragma unroll 1
    for (int m = 0; m < 6; ++m) {
        MhdWave<double> q;
        if (!mhd_six_wave<double, true>(s, six, gg, m, q, R[2 + m])) return false;
        mhd_wave_dU<double>(s, gg, q, R[2 + m]);
        const double db = (q.rho - s.beta * q.p) * s.ip;
        double *x = X[2 + m], *a = A[2 + m];
        x[0] = (gam * q.rho * ir - q.p * s.ip) * gm1i + db;
        x[4] = -(db * s.W + s.beta * q.u[0]);
        a[0] = q.rho;
        a[4] = q.p;
        for (int k = 0; k < 3; ++k) {
            x[1 + k] = db * s.u[1 + k] + s.beta * q.u[1 + k];
            x[5 + k] = db * s.b[1 + k] + s.beta * q.b[1 + k];
            a[1 + k] = (q.u[1 + k] - wrot[1 + k] * q.u[0]) * s.iW;
            a[5 + k] = R[2 + m][5 + k];
        }
        if (cluster) {   // the wave's coefficients in the y_a
            const double ga = -a[5] * __drcp_rn(1.0 - s.v1 * s.v1);
            for (int k = 0; k < 4; ++k) S[k][m] = a[1 + k];
            S[4][m] = a[6] - ga * s.v1 * wrot[2];
            S[5][m] = a[7] - ga * s.v1 * wrot[3];
        }
    }
    double lhat = 0.0;
    int msel = 0;
    for (int m = 0; m < 8; ++m) {
        const double v = fabs(jt + Lk * lam[m]);
        if (v > lhat) { lhat = v; msel = m; }
    }
    const double sg = (jt + Lk * lam[msel]) >= 0.0 ? 1.0 : -1.0;
    hl = 0.5 * lhat;
    MhdClusters cl;
    if (cluster) {
        mhd_clusters(gam, wrot, lam, S, R, X, A, cl);
        mhd_turn(cl, R, true);   // the dissipation takes the canonical waves
    }
    for (int k = 0; k < NS; ++k)
        for (int b = 0; b < 8; ++b) gTV[k][b] = 0.0;
    for (int b = 0; b < 8; ++b) Rz[b] = 0.0;
    double Rb[8][8], zeta = 0.0;
#pragma unroll 1
    for (int m = 0; m < 8; ++m) {
        double Vt[NS], gVt[NS], scale = 0.0, qm = 0.0;
        for (int k = 0; k < NS; ++k) {
            double acc = 0.0;
            for (int a = 0; a < 8; ++a) {
                const double t = R[m][a] * TV[k][a];
                acc += t;
                if (k == OFF || k == OFF + 1) scale += fabs(t);
            }
            Vt[k] = acc;
        }
        for (int b = 0; b < 8; ++b) qm += R[m][b] * lrot[b];
        double vminus, vplus;
        if constexpr (WW == 5) weno5_lr<double>(Vt[0], Vt[1], Vt[2], Vt[3], Vt[4], Vt[5], ph.eps, vminus, vplus);
        else weno3_lr<double>(Vt[0], Vt[1], Vt[2], Vt[3], ph.eps, vminus, vplus);
        const double jw = vplus - vminus, jump = Vt[OFF + 1] - Vt[OFF];
        const int sj = fabs(jump) <= ph.sign_tol * scale ? 0 : sgn_d(jump);
        const bool y = sgn_d(jw) == sj;
        const double z = y ? jw : 0.0;
        zeta += qm * z;
        for (int b = 0; b < 8; ++b) {
            Rz[b] += R[m][b] * z;
            Rb[m][b] = -hl * lrot[b] * z;
        }
        if (!y) continue;
        weno_jump_vjp<WW>(Vt, ph.eps, -hl * qm, gVt);
        for (int k = 0; k < NS; ++k)
            for (int b = 0; b < 8; ++b) {
                gTV[k][b] += R[m][b] * gVt[k];
                Rb[m][b] += gVt[k] * TV[k][b];
            }
    }
    const double glam = -0.5 * sg * Lk * zeta;
    // coefficients of a_n^T G' a_m (cG[m][n]) and a_n^T K' a_m (cK[m][n]); first cG[m][n] =
    // dJ/dc_nm = r_n . Rbar_m
    double cG[8][8], cK[8][8], y1[8], eta[2] = {0.0, 0.0};
#pragma unroll 1
    for (int m = 0; m < 8; ++m)
        for (int n = 0; n < 8; ++n) {
            double P = 0.0;
            for (int b = 0; b < 8; ++b) P += R[n][b] * Rb[m][b];
            cG[m][n] = P;
            cK[m][n] = 0.0;
        }
    double Q[6][6];
    if (cluster) {
        // the rotations within the clusters, in reverse
        double gin[6][6];
        for (int l = 0; l < 6; ++l)
            for (int k = 0; k < 6; ++k) Q[l][k] = gin[l][k] = 0.0;
#pragma unroll 1
        for (int t = 0; t < 6; ++t) {
            const int f = cl.from[t];
            double y[6], a5 = 0.0;
            for (int q = f; q < cl.to[t]; ++q) a5 += cl.Th[q][t] * A[2 + q][5];
            for (int j = t - 1; j >= f; --j) {
                double acc = cG[2 + t][2 + j] - cG[2 + j][2 + t];
                for (int jj = j + 1; jj < t; ++jj) acc -= cl.Ec[cl.ii[jj]][j] * y[jj];
                y[j] = acc * __drcp_rn(cl.Ec[cl.ii[j]][j]);
            }
            for (int j = f; j < t; ++j) {
                const int i = cl.ii[j];
                for (int n = 0; n < 6; ++n) {
                    if (n < f || n >= cl.to[t]) gin[t][n] -= y[j] * cl.Ec[i][n];
                    else if (n <= j) gin[t][n] += 0.5 * y[j] * cl.Ec[i][n];
                }
                for (int l = i + 1; l < 6; ++l) Q[l][i] -= y[j] * cl.Ec[l][t];
                eta[0] -= y[j] * a5 * cl.L4[i];
                eta[1] -= y[j] * a5 * cl.L5[i];
            }
        }
        for (int m = 0; m < 6; ++m)
            for (int n = 0; n < 6; ++n) {
                const bool in = n >= cl.from[m] && n < cl.to[m];
                cG[2 + m][2 + n] = (in ? -0.5 : 1.0) * cG[2 + m][2 + n] + gin[m][n];
            }
        // back to the resolved waves, whose speeds the other terms divide by
        mhd_turn(cl, R, false);
        mhd_turn(cl, Rb, false);
        mhd_turn(cl, cG, false);
#pragma unroll 1
        for (int m = 0; m < 8; ++m) {
            double o[6];
            for (int n = 0; n < 6; ++n) {
                double acc = 0.0;
                for (int q = cl.from[n]; q < cl.to[n]; ++q) acc += cl.Th[n][q] * cG[m][2 + q];
                o[n] = acc;
            }
            for (int n = 0; n < 6; ++n) cG[m][2 + n] = o[n];
        }
    }
    for (int b = 0; b < 8; ++b) {
        double acc = Rb[1][b];
        for (int m = 1; m < 8; ++m) acc -= cG[m][1] * X[m][b];
        y1[b] = sd * acc;
    }
#pragma unroll 1
    for (int m = 0; m < 8; ++m)
        for (int n = 0; n < 8; ++n) {
            const double P = cG[m][n];
            if (m < 2) {
                cG[m][n] = n == m ? -0.5 * P : 0.0;
            } else if (n < 2) {
                cG[m][n] = -P;
            } else if (cluster && n - 2 >= cl.from[m - 2] && n - 2 < cl.to[m - 2]) {
                if (n == m && m == msel) {
                    cK[m][n] = glam;
                    cG[m][n] -= lam[m] * glam;
                }
            } else if (n != m) {
                const double K = P * __drcp_rn(lam[m] - lam[n]);
                cK[m][n] = K;
                cG[m][n] = -lam[m] * K;
            } else {
                cK[m][n] = m == msel ? glam : 0.0;
                cG[m][n] = -0.5 * P - lam[m] * cK[m][n];
            }
        }
    if (cluster) {
        // L^-1 G_y' L^-T: its part in G' and in the divergence direction
        const double iv = __drcp_rn(1.0 - s.v1 * s.v1);
        double d[6];
        for (int i = 0; i < 6; ++i) {
            double acc = 0.0;
            for (int m = 0; m < 6; ++m) acc += cl.E[i][m] * A[2 + m][5];
            d[i] = -acc * iv;
        }
#pragma unroll 1
        for (int n = 0; n < 6; ++n) {
            double kap = 0.0;
            for (int l = 0; l < 6; ++l) {
                double t = 0.0;   // sum_i Q[l][i] E[i][n]
                for (int i = 0; i < l; ++i) {
                    t += Q[l][i] * cl.E[i][n];
                    kap -= Q[l][i] * d[i] * cl.E[l][n];
                }
                kap -= t * d[l];
                for (int m = 0; m < 6; ++m) cG[2 + n][2 + m] += t * cl.E[l][m];
            }
            for (int b = 0; b < 8; ++b) y1[b] += kap * X[2 + n][b];
        }
    }
    double g[8] = {0, 0, 0, 0, 0, 0, 0, 0}, pp[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    if (msel < 2) g[1] += glam;   // lambda = v_1
#pragma unroll 1
    for (int m = 0; m < 8; ++m) {
        // adjoints of U_w' a_m, V_w' a_m and F~_w' a_m
        double aU[8], aV[8], aF[8];
        for (int b = 0; b < 8; ++b) {
            aU[b] = Rb[m][b];
            aV[b] = aF[b] = 0.0;
        }
        for (int n = 0; n < 8; ++n) {
            const double gx = cG[n][m], gr = cG[m][n] + cK[n][m] * lam[n], kf = cK[m][n];
            for (int b = 0; b < 8; ++b) {
                aU[b] += gx * X[n][b];
                aV[b] += gr * R[n][b];
                aF[b] += kf * X[n][b];
            }
        }
        dual wd[8], gd[8];
        for (int k = 0; k < 8; ++k) wd[k] = dual(wrot[k], A[m][k]);
        mhd_UFV_grad<dual>(gam, wd, aU, aF, aV, gd);
        for (int k = 0; k < 8; ++k) {
            g[k] += gd[k].d;
            pp[k] += aF[k] * A[m][5];   // the Powell column Phi'(V) dB_1
        }
    }
    const double *v = wrot + 1, *B = wrot + 5;
    const double iW2 = s.iW * s.iW, vB = v[0] * B[0] + v[1] * B[1] + v[2] * B[2];
    for (int k = 0; k < 3; ++k) {
        double av = pp[4] * B[k] + pp[5 + k], aB = pp[4] * v[k];
        for (int jj = 0; jj < 3; ++jj) {
            av += pp[1 + jj] * (-2.0 * B[jj] * v[k] + (jj == k ? vB : 0.0) + v[jj] * B[k]);
            aB += pp[1 + jj] * ((jj == k ? iW2 : 0.0) + v[jj] * v[k]);
        }
        g[1 + k] += av;
        g[5 + k] += aB;
    }
    // the divergence wave's own direction dB = e_1 - v_1 v
    {
        double q[3];
        const double mB = y1[1] * B[0] + y1[2] * B[1] + y1[3] * B[2], mv = y1[1] * v[0] + y1[2] * v[1] + y1[3] * v[2];
        for (int k = 0; k < 3; ++k)
            q[k] = 2.0 * B[k] * mv - v[k] * mB - vB * y1[1 + k] + y1[4] * (2.0 * B[k] - B[k] * iW2 - vB * v[k]) +
                   y1[5 + k];
        g[1] -= 2.0 * v[0] * q[0] + v[1] * q[1] + v[2] * q[2];
        g[2] -= v[0] * q[1];
        g[3] -= v[0] * q[2];
    }
    if (cluster) {   // h_k = v_1 v_k / (1 - v_1^2)
        const double iv = __drcp_rn(1.0 - v[0] * v[0]), e = (eta[0] * v[1] + eta[1] * v[2]) * iv;
        g[1] += e * (1.0 + v[0] * v[0]) * iv;
        g[2] += eta[0] * v[0] * iv;
        g[3] += eta[1] * v[0] * iv;
    }
    for (int k = 0; k < 8; ++k) gw[k] = g[k];
    return true;
}

template <int WW>
__device__ __forceinline__ void mhd_diss_vjp(const Phys &ph, const double wrot[8], double Lk, double jt,
                                             const double lrot[8], const double TV[][8], double gTV[][8], double gw[8],
                                             double Rz[8], double &hl)
{
    if (!mhd_diss_vjp_waves<WW>(ph, wrot, Lk, jt, lrot, TV, gTV, gw, Rz, hl))
        mhd_diss_vjp_gram<WW>(ph, wrot, Lk, jt, lrot, TV, gTV, gw, Rz, hl);
}

}  // namespace esmm

// esmm_adjoint.cu -- vector-Jacobian products of the right-hand side and of
// the SSP-RK3 step (gradients of a final-time functional
// with respect to the initial data).
//
// The map differentiated is one time step with its mesh velocity xdot and
// time step dt held at their recorded values (the mesh monitor's maximum and
// the movement limiter's minimum are not differentiable), and with the sign
// switch Y and the lambda^ maximum frozen at their forward selection.  With
// xdot fixed the metrics and J are independent of the state, so the adjoint
// runs through the conserved state only:
//   mu (adjoint of dU/dt)  ->  lambda_F = mu_{L+1} - mu_L per interface
//   -> per pair / per interface: reverse sweeps of the two-point flux (log
//      means and averages) and of the ES dissipation (eigenvectors, WENO weights)
//   -> per node: gather, chain rule to the primitives, and the implicit-
//      function adjoint of the Newton recovery, lambda_U = (dU/dw)^-T lambda_w
//   -> lambda_cons += lambda_U / J (ghost nodes add into their source node).
#include <cuda_runtime.h>

#include "esmm_flux.cuh"
#include "esmm_vjp.cuh"

namespace esmm {

namespace {

constexpr int NQA = 7;      // adjoint node quantities: beta, u_x, u_y, W, ln rho, ln beta, rho
constexpr int NSMAX = 6;    // stencil nodes of WENO5
// contributions of one interface: lambda_V of the stencil nodes [NSMAX][4], then
// rho_0, rho_1, ln rho_0, ln rho_1 of its two nodes, and beta, u_x, u_y (the same
// for both nodes)
constexpr int NGI = NSMAX * 4 + 7;
static_assert(2 * NGI == ADJ_G_PER_NODE, "the interface contributions' buffer");

__device__ __forceinline__ double mu_at(const Geom &g, const double *mu, int i, int j, int a)
{
    if (i < 0 || i >= g.nx || j < 0 || j >= g.ny) return 0.0;
    return mu[(long long)a * g.N + (long long)j * g.nx + i];
}

// lambda_F of the interface whose left node is (i, j) in direction dir
__device__ __forceinline__ void lambda_face(const Geom &g, const double *mu, int i, int j, int dir, double lf[4])
{
    int i1 = i + (dir == 0), j1 = j + (dir == 1);
#pragma unroll
    for (int a = 0; a < 4; ++a) lf[a] = mu_at(g, mu, i1, j1, a) - mu_at(g, mu, i, j, a);
}

__device__ __forceinline__ NodeV<double> node_value(const Geom &g, const double *q, long long c)
{
    return load_node<double>(g, q, nullptr, c);
}

// Adjoint of ec_pair: lp the adjoint of its four components; gl, gr receive the
// adjoints of the 7 node quantities of the two nodes.
__device__ __forceinline__ void ec_pair_vjp(const NodeV<double> &l, const NodeV<double> &r, double mt, double mx,
                                            double my, double gm1inv, double thr, const double lp[4], double gl[NQA],
                                            double gr[NQA])
{
    double rln, irln, bln, ibln;
    logmean2<double>(l.rho, r.rho, thr, rln, irln);
    logmean2<double>(l.beta, r.beta, thr, bln, ibln);
    const double rm = 0.5 * (l.rho.v + r.rho.v), bm = 0.5 * (l.beta.v + r.beta.v), W = 0.5 * (l.W + r.W);
    const double ux = 0.5 * (l.ux + r.ux), uy = 0.5 * (l.uy + r.uy);
    const double usq = ux * ux + uy * uy, Lam = W * W - usq, alpha0 = 1.0 + gm1inv * ibln;
    const double ibm = __drcp_rn(bm), pm = rm * ibm, rinv = __drcp_rn(Lam * W), iLam = rinv * W, iW = rinv * Lam;
    const double A = alpha0 * rln, UE = (A * W * W + pm * usq) * iLam, un = mx * ux + my * uy;
    const double Es = W * (A + pm) * un * iLam, cm = (mt * (UE + pm) + Es) * iW;
    // reverse
    const double gcm = lp[1] * ux + lp[2] * uy, gc = gcm * iW;
    double gux = lp[1] * cm, guy = lp[2] * cm, gpm = lp[1] * mx + lp[2] * my + gc * mt, gW = -gc * cm;
    const double gUE = (lp[3] + gc) * mt, gEs = lp[3] + gc;
    double grln = lp[0] * (mt * W + un), gun = lp[0] * rln;
    gW += lp[0] * rln * mt;
    const double e1 = gUE * iLam, e2 = gEs * iLam;
    double gA = e1 * W * W + e2 * W * un;
    gW += e1 * 2.0 * A * W + e2 * (A + pm) * un;
    gpm += e1 * usq + e2 * W * un;
    double gusq = e1 * pm;
    gun += e2 * W * (A + pm);
    const double gLam = -(e1 * UE + e2 * Es);
    gW += 2.0 * W * gLam;
    gusq -= gLam;
    gux += 2.0 * ux * gusq + mx * gun;
    guy += 2.0 * uy * gusq + my * gun;
    grln += gA * alpha0;
    const double gb = gpm * ibm;
    const double hb = -0.5 * gb * pm, hr = 0.5 * gb;
    gl[0] = gr[0] = hb;
    gl[1] = gr[1] = 0.5 * gux;
    gl[2] = gr[2] = 0.5 * guy;
    gl[3] = gr[3] = 0.5 * gW;
    gl[4] = gr[4] = gl[5] = gr[5] = 0.0;
    gl[6] = gr[6] = hr;
    logmean_vjp(l.rho.v, r.rho.v, l.rho.l, r.rho.l, thr, grln, gl[6], gr[6], gl[4], gr[4]);
    logmean_vjp(l.beta.v, r.beta.v, l.beta.l, r.beta.l, thr, -gA * rln * gm1inv * ibln * ibln, gl[0], gr[0], gl[5], gr[5]);
}

// Adjoint contributions of the pair fluxes anchored at A: the pair (A, A+n)
// enters the interfaces A + s (s < n) with weight alpha_{p,n}, so its adjoint
// is alpha_n sum_s lambda_F(A + s).
template <int P>
__global__ void __launch_bounds__(128) k_pairs_vjp(ProbArg pa, Phys ph, const double *__restrict__ q,
                                                   const double *__restrict__ mu, double *__restrict__ Gp, int dir)
{
    ProbDesc D;
    long long lb;
    locate(pa, D, lb);
    const Geom &g = D.g;
    q += (long long)NQ * D.op;
    mu += 4 * D.on;
    Gp += (long long)2 * PMAX * 2 * NQA * D.op;
    const int nd = dir == 0 ? g.nx : g.ny, no = dir == 0 ? g.ny : g.nx;
    const long long idx = lb * blockDim.x + threadIdx.x;
    if (idx >= (long long)(nd + P) * no) return;
    int i, j;
    if (dir == 0) { j = (int)(idx / (nd + P)); i = (int)(idx % (nd + P)) - P; }
    else { i = (int)(idx % no); j = (int)(idx / no) - P; }
    const long long c0 = pidx(g, i, j);
    const long long sd = dir == 0 ? 1 : g.px;
    const double *Mt = q + (Q_MT0 + dir) * g.P;
    const double *Mx = q + (Q_M00 + 2 * dir) * g.P;
    const double *My = q + (Q_M01 + 2 * dir) * g.P;
    const double gm1inv = 1.0 / (ph.gamma - 1.0);
    const NodeV<double> nl = node_value(g, q, c0);
    const int A = dir == 0 ? i : j;
    for (int n = 1; n <= P; ++n) {
        double lp[4] = {0.0, 0.0, 0.0, 0.0};
        for (int s = 0; s < n; ++s) {
            int L = A + s;
            if (L < -1 || L > nd - 1) continue;
            double lf[4];
            lambda_face(g, mu, dir == 0 ? L : i, dir == 0 ? j : L, dir, lf);
#pragma unroll
            for (int a = 0; a < 4; ++a) lp[a] += lf[a];
        }
#pragma unroll
        for (int a = 0; a < 4; ++a) lp[a] *= ph.alpha[n - 1];
        const long long cr = c0 + n * sd;
        const NodeV<double> nr = node_value(g, q, cr);
        double gl[NQA], gr[NQA];
        ec_pair_vjp(nl, nr, 0.5 * (Mt[c0] + Mt[cr]), 0.5 * (Mx[c0] + Mx[cr]), 0.5 * (My[c0] + My[cr]), gm1inv,
                    ph.ln_thr, lp, gl, gr);
        double *o = Gp + ((long long)(dir * PMAX + (n - 1)) * 2) * NQA * g.P + c0;
#pragma unroll
        for (int jq = 0; jq < NQA; ++jq) {
            o[jq * g.P] = gl[jq];
            o[(NQA + jq) * g.P] = gr[jq];
        }
    }
}

// Adjoint of the ES dissipation at one interface: F = F_EC - diss, so the
// objective's part is -lambda_F . diss.  Reverse sweep through the WENO jumps, the
// projections on the scaled eigenvectors (eigen_rhd) and the interface state; Y
// and the lambda^ maximum keep their forward selection.  Bound: the FP64 pipe, at
// about three times the forward dissipation.  Measured (GB300, 200 x 200 nodes,
// the whole vector-Jacobian product): 0.53 ms, against 15.5 ms with dual numbers
// seeded at each of the 38 stencil values and of the pair's 14 in turn.
template <int WW>
__global__ void __launch_bounds__(128) k_iface_vjp(ProbArg pa, Phys ph, const double *__restrict__ q,
                                                   const double *__restrict__ mu, double *__restrict__ G, int dir)
{
    constexpr int NS = WW + 1, OFF = (WW - 1) / 2;
    ProbDesc D;
    long long lb;
    locate(pa, D, lb);
    const Geom &g = D.g;
    q += (long long)NQ * D.op;
    mu += 4 * D.on;
    G += (long long)2 * NGI * D.op;
    const int nd = dir == 0 ? g.nx : g.ny, no = dir == 0 ? g.ny : g.nx;
    const long long idx = lb * blockDim.x + threadIdx.x;
    if (idx >= (long long)(nd + 1) * no) return;
    int i, j;
    if (dir == 0) { j = (int)(idx / (nd + 1)); i = (int)(idx % (nd + 1)) - 1; }
    else { i = (int)(idx % no); j = (int)(idx / no) - 1; }
    const long long c0 = pidx(g, i, j);
    const long long sd = dir == 0 ? 1 : g.px;
    const long long c1 = c0 + sd;
    double lf[4];
    lambda_face(g, mu, i, j, dir, lf);
    const double *Mt = q + (Q_MT0 + dir) * g.P;
    const double *Mx = q + (Q_M00 + 2 * dir) * g.P;
    const double *My = q + (Q_M01 + 2 * dir) * g.P;
    const double nvx = 0.5 * (Mx[c0] + Mx[c1]), nvy = 0.5 * (My[c0] + My[c1]), jt = 0.5 * (Mt[c0] + Mt[c1]);
    // forward: the interface state and the scaled eigenvectors (as es_dissipation, eigen_rhd)
    const double n2 = nvx * nvx + nvy * nvy, iLk = rsqrt(n2), Lk = n2 * iLk, nx = nvx * iLk, ny = nvy * iLk;
    const double r0 = q[Q_RHO * g.P + c0], r1 = q[Q_RHO * g.P + c1];
    const double l0 = q[Q_LNR * g.P + c0], l1 = q[Q_LNR * g.P + c1];
    double rho, irho;
    logmean<double, double>(r0, r1, l0, l1, ph.ln_thr, rho, irho);
    const double ux = 0.5 * (q[Q_UX * g.P + c0] + q[Q_UX * g.P + c1]);
    const double uy = 0.5 * (q[Q_UY * g.P + c0] + q[Q_UY * g.P + c1]);
    const double ib = __drcp_rn(q[Q_BETA * g.P + c0] + q[Q_BETA * g.P + c1]), p = (r0 + r1) * ib;
    const double w2 = 1.0 + ux * ux + uy * uy, iW = rsqrt(w2), W = w2 * iW;
    const double vx = ux * iW, vy = uy * iW, vn = nx * vx + ny * vy, vt = -ny * vx + nx * vy;
    const double gam = ph.gamma, gm1i = ph.gm1i, gg = gam * gm1i, c1g = gg;
    const double W2 = W * W, iW2 = __drcp_rn(W2), v2 = 1.0 - iW2, W3 = W2 * W, W4 = W2 * W2;
    const double ip = __drcp_rn(p), ir = __drcp_rn(rho), rh = rho + gg * p, irh = __drcp_rn(rh);
    const double cc2 = gam * p * irh, icc = rsqrt(cc2), cc = cc2 * icc;
    const double D0 = 1.0 - v2 * cc2, X = D0 - vn * vn * (1.0 - cc2), Y = iW2 * X, idisc = rsqrt(Y), disc = Y * idisc;
    const double den = __drcp_rn(D0);
    const double Q = rh * W2, beta = rho * ip, un = W * vn, ut = W * vt;
    double lam[2];
    lam[0] = (vn * (1.0 - cc2) - cc * disc) * den;
    lam[1] = (vn * (1.0 - cc2) + cc * disc) * den;
    const double sp0 = jt + Lk * lam[0], sp1 = jt + Lk * lam[1];
    const int sel = fabs(sp0) >= fabs(sp1) ? 0 : 1;
    const double spl = sel ? sp1 : sp0, lhat = fabs(spl);
    double dU[4][4], s[4];
    dU[0][1] = W; dU[1][1] = W2 * vn; dU[2][1] = W2 * vt; dU[3][1] = W2;
    s[1] = rsqrt(gg * W * ir);
    dU[0][2] = rho * W3 * vt;
    dU[1][2] = 2.0 * rh * W4 * vn * vt;
    dU[2][2] = rh * (2.0 * W4 * vt * vt + W2);
    dU[3][2] = 2.0 * rh * W4 * vt;
    const double sh = 1.0 + W2 * vt * vt;
    s[2] = rsqrt(rh * beta * W3 * sh);
    double a_[2], dvn_[2], dvt_[2], vdv_[2], drho_[2], dV_[2][4];
#pragma unroll
    for (int side = 0; side < 2; ++side) {
        const int m = side ? 3 : 0;
        const double l = lam[side], a = __drcp_rn((l - vn) * Q);
        const double dvn = (1.0 - vn * l) * a, dvt = -l * vt * a, vdv = vn * dvn + vt * dvt;
        const double drho = rho * dvn * a * Q - rho * W2 * vdv, h1 = drho + gg, dW = W3 * vdv;
        dU[0][m] = W * drho + rho * dW;
        dU[1][m] = W2 * vn * h1 + rh * (2.0 * W4 * vn * vdv + W2 * dvn);
        dU[2][m] = W2 * vt * h1 + rh * (2.0 * W4 * vt * vdv + W2 * dvt);
        dU[3][m] = W2 * h1 - 1.0 + rh * 2.0 * W4 * vdv;
        const double dbeta = drho * ip - beta * ip;
        dV_[side][0] = drho * ir + (drho * ir - ip) * gm1i + dbeta;
        dV_[side][1] = dbeta * un + beta * (W * dvn + vn * dW);
        dV_[side][2] = dbeta * ut + beta * (W * dvt + vt * dW);
        dV_[side][3] = -(dbeta * W + beta * dW);
        s[m] = rsqrt(dU[0][m] * dV_[side][0] + dU[1][m] * dV_[side][1] + dU[2][m] * dV_[side][2] + dU[3][m] * dV_[side][3]);
        a_[side] = a; dvn_[side] = dvn; dvt_[side] = dvt; vdv_[side] = vdv; drho_[side] = drho;
    }
    // projections and jumps; then their adjoints
    NodeStencil<double, QGet> st{{q, g.P, c0, sd, OFF}};
    double TV[NS][4], aT[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int k = 0; k < NS; ++k) {
        double V[4];
        st.V(k, c1g, gm1i, V);
        TV[k][0] = V[0];
        TV[k][1] = nx * V[1] + ny * V[2];
        TV[k][2] = -ny * V[1] + nx * V[2];
        TV[k][3] = V[3];
        if (k == OFF || k == OFF + 1)
#pragma unroll
            for (int a = 0; a < 4; ++a) aT[a] += fabs(TV[k][a]);
    }
    const double lrot[4] = {lf[0], nx * lf[1] + ny * lf[2], -ny * lf[1] + nx * lf[2], lf[3]};
    const double hl = 0.5 * lhat;
    double gU[4][4], gs[4], glh = 0.0, gTV[NS][4];
#pragma unroll
    for (int k = 0; k < NS; ++k)
#pragma unroll
        for (int a = 0; a < 4; ++a) gTV[k][a] = 0.0;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        double P[NS], Vt[NS], gVt[NS];   // dU_m . TV_k, and the projections s_m P_k
#pragma unroll
        for (int k = 0; k < NS; ++k) {
            P[k] = dU[0][m] * TV[k][0] + dU[1][m] * TV[k][1] + dU[2][m] * TV[k][2] + dU[3][m] * TV[k][3];
            Vt[k] = s[m] * P[k];
        }
        double vminus, vplus;
        if (WW == 5) weno5_lr<double>(Vt[0], Vt[1], Vt[2], Vt[3], Vt[NS - 2], Vt[NS - 1], ph.eps, vminus, vplus);
        else weno3_lr<double>(Vt[0], Vt[1], Vt[2], Vt[3], ph.eps, vminus, vplus);
        const double jw = vplus - vminus, jump = Vt[OFF + 1] - Vt[OFF];
        const double scale = s[m] * (fabs(dU[0][m]) * aT[0] + fabs(dU[1][m]) * aT[1] + fabs(dU[2][m]) * aT[2] +
                                     fabs(dU[3][m]) * aT[3]);
        const int sj = fabs(jump) <= ph.sign_tol * scale ? 0 : sgn_d(jump);
        const double jy = sgn_d(jw) == sj ? jw : 0.0;
        const double qm = lrot[0] * dU[0][m] + lrot[1] * dU[1][m] + lrot[2] * dU[2][m] + lrot[3] * dU[3][m];
        glh -= 0.5 * qm * s[m] * jy;
        gs[m] = -hl * qm * jy;
#pragma unroll
        for (int a = 0; a < 4; ++a) gU[a][m] = -hl * lrot[a] * s[m] * jy;
        if (sgn_d(jw) != sj) continue;   // Y = 0
        weno_jump_vjp<WW>(Vt, ph.eps, -hl * qm * s[m], gVt);
#pragma unroll
        for (int k = 0; k < NS; ++k) {
            gs[m] += gVt[k] * P[k];
            const double gk = gVt[k] * s[m];
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                gTV[k][a] += gk * dU[a][m];
                gU[a][m] += gk * TV[k][a];
            }
        }
    }
    double *o = G + (long long)(dir * NGI) * g.P + c0;
#pragma unroll
    for (int k = 0; k < NS; ++k) {
        o[(4 * k) * g.P] = gTV[k][0];
        o[(4 * k + 1) * g.P] = nx * gTV[k][1] - ny * gTV[k][2];
        o[(4 * k + 2) * g.P] = ny * gTV[k][1] + nx * gTV[k][2];
        o[(4 * k + 3) * g.P] = gTV[k][3];
    }
    // reverse of eigen_rhd
    double gW = 0.0, gW2 = 0.0, gW3 = 0.0, gW4 = 0.0, grho = 0.0, grh = 0.0, gvn = 0.0, gvt = 0.0, gbeta = 0.0,
           gip = 0.0, gir = 0.0, gun = 0.0, gut = 0.0, gQ = 0.0, gl_[2] = {0.0, 0.0};
    gl_[sel] += (spl >= 0.0 ? Lk : -Lk) * glh;
    {   // entropy wave
        gW += gU[0][1];
        gW2 += gU[1][1] * vn + gU[2][1] * vt + gU[3][1];
        gvn += gU[1][1] * W2;
        gvt += gU[2][1] * W2;
        const double ga = -0.5 * s[1] * s[1] * s[1] * gs[1];
        gW += ga * gg * ir;
        gir += ga * gg * W;
    }
    {   // shear wave
        const double a0 = gU[0][2], a1 = gU[1][2], a2 = gU[2][2], a3 = gU[3][2];
        grho += a0 * W3 * vt;
        gW3 += a0 * rho * vt;
        const double e = 2.0 * (a1 * vn + a2 * vt + a3);
        grh += e * W4 * vt + a2 * W2;
        gW4 += e * rh * vt;
        gvn += a1 * 2.0 * rh * W4 * vt;
        gvt += a0 * rho * W3 + 2.0 * rh * W4 * (a1 * vn + 2.0 * a2 * vt + a3);
        gW2 += a2 * rh;
        const double ga = -0.5 * s[2] * s[2] * s[2] * gs[2];
        grh += ga * beta * W3 * sh;
        gbeta += ga * rh * W3 * sh;
        gW3 += ga * rh * beta * sh;
        const double gsh = ga * rh * beta * W3;
        gW2 += gsh * vt * vt;
        gvt += gsh * 2.0 * W2 * vt;
    }
#pragma unroll
    for (int side = 0; side < 2; ++side) {
        const int m = side ? 3 : 0;
        const double l = lam[side], a = a_[side], dvn = dvn_[side], dvt = dvt_[side], vdv = vdv_[side],
                     drho = drho_[side], h1 = drho + gg, dW = W3 * vdv, dbeta = drho * ip - beta * ip;
        const double gN = -0.5 * s[m] * s[m] * s[m] * gs[m];
        double u[4], V[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            u[k] = gU[k][m] + gN * dV_[side][k];
            V[k] = gN * dU[k][m];
        }
        double gdb = -V[3] * W + V[2] * ut + V[1] * un + V[0], gdW = (V[2] * vt + V[1] * vn - V[3]) * beta;
        gW += -V[3] * dbeta + (V[2] * dvt + V[1] * dvn) * beta;
        gbeta += -V[3] * dW + V[2] * (W * dvt + vt * dW) + V[1] * (W * dvn + vn * dW);
        gut += V[2] * dbeta;
        gun += V[1] * dbeta;
        double gdvt = V[2] * beta * W, gdvn = V[1] * beta * W;
        gvt += V[2] * beta * dW;
        gvn += V[1] * beta * dW;
        double gdr = V[0] * ir * (1.0 + gm1i);
        gir += V[0] * drho * (1.0 + gm1i);
        gip -= V[0] * gm1i;
        gdr += gdb * ip;
        gip += gdb * (drho - beta);
        gbeta -= gdb * ip;
        const double e = u[1] * vn + u[2] * vt + u[3], f = u[1] * dvn + u[2] * dvt;
        gW2 += e * h1 + f * rh;
        double gh1 = e * W2;
        grh += 2.0 * W4 * vdv * e + W2 * f;
        gW4 += 2.0 * rh * vdv * e;
        double gvdv = 2.0 * rh * W4 * e;
        const double hv = W2 * h1 + 2.0 * rh * W4 * vdv;
        gvt += u[2] * hv;
        gvn += u[1] * hv;
        gdvt += u[2] * rh * W2;
        gdvn += u[1] * rh * W2;
        gW += u[0] * drho;
        gdr += u[0] * W + gh1;
        grho += u[0] * dW;
        gdW += u[0] * rho;
        gW3 += gdW * vdv;
        gvdv += gdW * W3;
        const double aQ = a * Q;
        grho += gdr * (dvn * aQ - W2 * vdv);
        gdvn += gdr * rho * aQ;
        double ga = gdr * rho * dvn * Q;
        gQ += gdr * rho * dvn * a;
        gW2 -= gdr * rho * vdv;
        gvdv -= gdr * rho * W2;
        gvn += gvdv * dvn;
        gdvn += gvdv * vn;
        gvt += gvdv * dvt;
        gdvt += gvdv * vt;
        gl_[side] -= gdvt * vt * a;
        gvt -= gdvt * l * a;
        ga -= gdvt * l * vt;
        gvn -= gdvn * l * a;
        gl_[side] -= gdvn * vn * a;
        ga += gdvn * (1.0 - vn * l);
        const double gaa = ga * a * a;
        gl_[side] -= gaa * Q;
        gvn += gaa * Q;
        gQ -= gaa * (l - vn);
    }
    const double gnm = gl_[0] * den, gnp = gl_[1] * den;
    const double gden = (gl_[0] * lam[0] + gl_[1] * lam[1]) * D0;
    double gc2 = -(gnm + gnp) * vn;
    gvn += (gnm + gnp) * (1.0 - cc2);
    const double gY = 0.5 * (gnp - gnm) * cc * idisc;
    gc2 += 0.5 * (gnp - gnm) * disc * icc;
    double giW2 = gY * X;
    const double gX = gY * iW2;
    const double gD0 = gX - gden * den * den;
    gvn -= 2.0 * vn * (1.0 - cc2) * gX;
    gc2 += vn * vn * gX - gD0 * v2;
    giW2 += gD0 * cc2;   // v2 = 1 - iW2
    double gp = gc2 * gam * irh;
    grh -= gc2 * cc2 * irh;
    gW2 -= giW2 * iW2 * iW2;
    gW += gun * vn + gut * vt;
    gvn += gun * W;
    gvt += gut * W;
    grh += gQ * W2;
    gW2 += gQ * rh;
    grho += gbeta * ip + grh - gir * ir * ir;
    gip += gbeta * rho;
    gp += gg * grh - gip * ip * ip;
    gW2 += 2.0 * W2 * gW4 + gW3 * W;
    gW += gW3 * W2 + 2.0 * W * gW2;
    // the interface state from the two nodes
    const double gvx = nx * gvn - ny * gvt, gvy = ny * gvn + nx * gvt;
    gW -= (gvx * ux + gvy * uy) * iW * iW;
    const double gux = gvx * iW + gW * ux * iW, guy = gvy * iW + gW * uy * iW;
    double g0 = gp * ib, g1 = g0, gl0 = 0.0, gl1 = 0.0;
    logmean_vjp(r0, r1, l0, l1, ph.ln_thr, grho, g0, g1, gl0, gl1);
    o += (long long)(NSMAX * 4) * g.P;
    o[0] = g0;
    o[g.P] = g1;
    o[2 * g.P] = gl0;
    o[3 * g.P] = gl1;
    o[4 * g.P] = -gp * p * ib;
    o[5 * g.P] = 0.5 * gux;
    o[6 * g.P] = 0.5 * guy;
}

// Per padded node: gather the pair and interface contributions, chain them to
// the primitives w = (rho, v_x, v_y, p), apply the recovery's adjoint
// lambda_U = (dU/dw)^-T lambda_w and add lambda_U / J into the source node.
__global__ void k_node_vjp(ProbArg pa, double gam, int p, int ww, const double *__restrict__ q,
                           const double *__restrict__ G, const double *__restrict__ Gp,
                           const double *__restrict__ J, double *__restrict__ lam)
{
    ProbDesc D;
    long long lb;
    locate(pa, D, lb);
    const Geom &g = D.g;
    long long t = lb * blockDim.x + threadIdx.x;
    if (t >= g.P) return;
    q += (long long)NQ * D.op;
    G += (long long)2 * NGI * D.op;
    Gp += (long long)2 * PMAX * 2 * NQA * D.op;
    J += D.on;
    lam += 4 * D.on;
    const int I = (int)(t % g.px) - GH, Jn = (int)(t / g.px) - GH;
    double lq[NQA] = {0, 0, 0, 0, 0, 0, 0}, lV[4] = {0, 0, 0, 0};
    const int NS = ww + 1, OFF = (ww - 1) / 2;
    for (int dir = 0; dir < 2; ++dir) {
        const int nd = dir == 0 ? g.nx : g.ny, no = dir == 0 ? g.ny : g.nx;
        const int pos = dir == 0 ? I : Jn, line = dir == 0 ? Jn : I;
        if (line < 0 || line >= no) continue;
        auto cidx = [&](int a) { return dir == 0 ? pidx(g, a, line) : pidx(g, line, a); };
        if (ww > 0)
            for (int k = 0; k < NS; ++k) {
                int L = pos - (k - OFF);
                if (L < -1 || L > nd - 1) continue;
                const double *o = G + (long long)(dir * NGI) * g.P + cidx(L);
                for (int a = 0; a < 4; ++a) lV[a] += o[(4 * k + a) * g.P];
                if (k != OFF && k != OFF + 1) continue;
                const int r = k - OFF;     // left or right node of the interface
                o += (long long)(NSMAX * 4) * g.P;
                lq[6] += o[r * g.P];
                lq[4] += o[(2 + r) * g.P];
                lq[0] += o[4 * g.P];
                lq[1] += o[5 * g.P];
                lq[2] += o[6 * g.P];
            }
        for (int n = 1; n <= p; ++n)
            for (int side = 0; side < 2; ++side) {
                int A = pos - side * n;
                if (A < -p || A > nd - 1) continue;
                long long ca = cidx(A);
                for (int jq = 0; jq < NQA; ++jq)
                    lq[jq] += Gp[((((long long)dir * PMAX + (n - 1)) * 2 + side) * NQA + jq) * g.P + ca];
            }
    }
    {   // V = (c + ln rho + ln beta/(Gamma-1) + beta, beta u, -beta W)
        const double b = q[Q_BETA * g.P + t];
        lq[0] += lV[0] + lV[1] * q[Q_UX * g.P + t] + lV[2] * q[Q_UY * g.P + t] - lV[3] * q[Q_W * g.P + t];
        lq[1] += lV[1] * b;
        lq[2] += lV[2] * b;
        lq[3] -= lV[3] * b;
        lq[4] += lV[0];
        lq[5] += lV[0] / (gam - 1.0);
    }
    // node quantities -> primitives
    double rho = q[Q_RHO * g.P + t], pr = q[Q_P * g.P + t], W = q[Q_W * g.P + t];
    double vx = q[Q_UX * g.P + t] / W, vy = q[Q_UY * g.P + t] / W;
    double W3 = W * W * W;
    double lw[4];
    lw[0] = lq[6] + lq[0] / pr + (lq[4] + lq[5]) / rho;
    lw[3] = -lq[0] * rho / (pr * pr) - lq[5] / pr;
    lw[1] = lq[1] * (W + vx * W3 * vx) + lq[2] * (vy * W3 * vx) + lq[3] * (W3 * vx);
    lw[2] = lq[1] * (vx * W3 * vy) + lq[2] * (W + vy * W3 * vy) + lq[3] * (W3 * vy);
    // dU/dw (rows D, m_x, m_y, E; columns rho, v_x, v_y, p)
    double g1 = gam / (gam - 1.0), rh = rho + g1 * pr, W2 = W * W, W4 = W2 * W2;
    double A[4][4] = {
        {W, rho * W3 * vx, rho * W3 * vy, 0.0},
        {W2 * vx, rh * (2.0 * W4 * vx * vx + W2), rh * 2.0 * W4 * vy * vx, g1 * W2 * vx},
        {W2 * vy, rh * 2.0 * W4 * vx * vy, rh * (2.0 * W4 * vy * vy + W2), g1 * W2 * vy},
        {W2, rh * 2.0 * W4 * vx, rh * 2.0 * W4 * vy, g1 * W2 - 1.0}};
    // solve A^T x = lw (Gaussian elimination with partial pivoting on M = A^T)
    double M[4][5];
    for (int r = 0; r < 4; ++r) {
        for (int c = 0; c < 4; ++c) M[r][c] = A[c][r];
        M[r][4] = lw[r];
    }
    for (int c = 0; c < 4; ++c) {
        int piv = c;
        for (int r = c + 1; r < 4; ++r)
            if (fabs(M[r][c]) > fabs(M[piv][c])) piv = r;
        if (piv != c)
            for (int k = 0; k < 5; ++k) { double tmp = M[c][k]; M[c][k] = M[piv][k]; M[piv][k] = tmp; }
        for (int r = c + 1; r < 4; ++r) {
            double f = M[r][c] / M[c][c];
            for (int k = c; k < 5; ++k) M[r][k] -= f * M[c][k];
        }
    }
    double xs[4];
    for (int r = 3; r >= 0; --r) {
        double acc = M[r][4];
        for (int k = r + 1; k < 4; ++k) acc -= M[r][k] * xs[k];
        xs[r] = acc / M[r][r];
    }
    long long src = data_src(g, I, Jn);
    double iJ = 1.0 / J[src];
    for (int a = 0; a < 4; ++a)
        if (xs[a] != 0.0) atomicAdd(lam + a * g.N + src, xs[a] * iJ);
}

// out = a x + b y over n values
__global__ void k_lincomb(long long n, double a, const double *__restrict__ x, double b, const double *__restrict__ y,
                          double *__restrict__ out)
{
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = a * x[i] + (y ? b * y[i] : 0.0);
}

// gradient with respect to the initial primitives: cons = J U(w), so
// lambda_w = J (dU/dw)^T lambda_cons
__global__ void k_prim_grad(ProbArg pa, double gam, const double *__restrict__ cons, const double *__restrict__ J,
                            const double *__restrict__ lam, double *__restrict__ out)
{
    ProbDesc D;
    long long lb;
    locate(pa, D, lb);
    const Geom &g = D.g;
    long long id = lb * blockDim.x + threadIdx.x;
    if (id >= g.N) return;
    cons += 4 * D.on;
    J += D.on;
    lam += 4 * D.on;
    out += 4 * D.on;
    double iJ = 1.0 / J[id];
    double rho, vx, vy, pr, W;
    cons2prim(gam, cons[id] * iJ, cons[g.N + id] * iJ, cons[2 * g.N + id] * iJ, cons[3 * g.N + id] * iJ, -1.0, rho,
              vx, vy, pr, W);
    double g1 = gam / (gam - 1.0), rh = rho + g1 * pr, W2 = W * W, W3 = W2 * W, W4 = W2 * W2;
    double A[4][4] = {
        {W, rho * W3 * vx, rho * W3 * vy, 0.0},
        {W2 * vx, rh * (2.0 * W4 * vx * vx + W2), rh * 2.0 * W4 * vy * vx, g1 * W2 * vx},
        {W2 * vy, rh * 2.0 * W4 * vx * vy, rh * (2.0 * W4 * vy * vy + W2), g1 * W2 * vy},
        {W2, rh * 2.0 * W4 * vx, rh * 2.0 * W4 * vy, g1 * W2 - 1.0}};
    for (int c = 0; c < 4; ++c) {
        double acc = 0.0;
        for (int r = 0; r < 4; ++r) acc += A[r][c] * lam[r * g.N + id];
        out[c * g.N + id] = J[id] * acc;
    }
}

}  // namespace

void launch_pairs_vjp(const LaunchDom &L, const Phys &ph, const double *q, const double *mu, double *Gp, int dir,
                      cudaStream_t st)
{
    if (ph.p == 1) k_pairs_vjp<1><<<L.nblk, L.bs, 0, st>>>(L.pa, ph, q, mu, Gp, dir);
    else if (ph.p == 2) k_pairs_vjp<2><<<L.nblk, L.bs, 0, st>>>(L.pa, ph, q, mu, Gp, dir);
    else k_pairs_vjp<3><<<L.nblk, L.bs, 0, st>>>(L.pa, ph, q, mu, Gp, dir);
}

void launch_iface_vjp(const LaunchDom &L, const Phys &ph, const double *q, const double *mu, double *G, int dir,
                      cudaStream_t st)
{
    if (ph.w == 5) k_iface_vjp<5><<<L.nblk, L.bs, 0, st>>>(L.pa, ph, q, mu, G, dir);
    else if (ph.w == 3) k_iface_vjp<3><<<L.nblk, L.bs, 0, st>>>(L.pa, ph, q, mu, G, dir);
}

void launch_node_vjp(const LaunchDom &L, double gam, int p, int w, const double *q, const double *G,
                     const double *Gp, const double *J, double *lam, cudaStream_t st)
{
    k_node_vjp<<<L.nblk, L.bs, 0, st>>>(L.pa, gam, p, w, q, G, Gp, J, lam);
}

void launch_lincomb(long long n, double a, const double *x, double b, const double *y, double *out, cudaStream_t st)
{
    k_lincomb<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, a, x, b, y, out);
}

void launch_prim_grad(const LaunchDom &L, double gam, const double *cons, const double *J, const double *lam,
                      double *out, cudaStream_t st)
{
    k_prim_grad<<<L.nblk, L.bs, 0, st>>>(L.pa, gam, cons, J, lam, out);
}

}  // namespace esmm

// esmm_flux.cuh -- the two flux kernels of one sweep direction:
//   k_pairs: every two-point EC flux F~_k(U_A, U_{A+n}) (Sec. 3.1), n = 1..p,
//            computed once per node pair and stored;
//   k_iface: the w-th order ES interface flux (eq. ESFlux_HO): the 2p-th order
//            combination of the stored pair fluxes (eq. ECFlux_O2p) minus the
//            WENO dissipation on scaled entropy variables, plus the metric
//            flux of the VCL (eq. MetricsFlux_O2p).
// One thread per node pair / interface, flattened over the sweep so that warps
// read consecutive nodes.
#pragma once

#include <type_traits>

#include "esmm_device.cuh"
#include "esmm_launch.h"

namespace esmm {

// One flux argument from the node arrays q (FP64) or from the FP32 copies q32 (float,
// with the FP64 rest of rho and beta for their jumps).
template <typename R>
__device__ __forceinline__ NodeV<R> load_node(const Geom &g, const double *__restrict__ q,
                                              const float *__restrict__ q32, long long c)
{
    NodeV<R> v;
    if constexpr (std::is_same<R, float>::value) {
        v.rho = lmv_f32(q[Q_RHO * g.P + c], q32[Q32_R * g.P + c], q32[Q32_LNR * g.P + c]);
        v.beta = lmv_f32(q[Q_BETA * g.P + c], q32[Q32_B * g.P + c], q32[Q32_LNB * g.P + c]);
        v.ux = q32[Q32_UX * g.P + c];
        v.uy = q32[Q32_UY * g.P + c];
        v.W = q32[Q32_W * g.P + c];
    } else {
        v.rho.v = q[Q_RHO * g.P + c];
        v.rho.l = q[Q_LNR * g.P + c];
        v.beta.v = q[Q_BETA * g.P + c];
        v.beta.l = q[Q_LNB * g.P + c];
        v.ux = q[Q_UX * g.P + c];
        v.uy = q[Q_UY * g.P + c];
        v.W = q[Q_W * g.P + c];
    }
    return v;
}

// The entropy variables (V_1, V_x, V_y, V_E) of one node (Sec. 2, B = 0)
// from beta, u, W, ln rho, ln beta: V_1 = Gamma/(Gamma-1) + ln rho +
// ln beta/(Gamma-1) + beta, (V_x, V_y) = beta u, V_E = -beta W.  Every
// stencil type below forms them with this one function, so a kernel that
// stores them per node gets the values a kernel forming them per interface
// gets: in FP64 and FP32 each operation is an explicitly rounded intrinsic,
// which leaves the compiler no choice of contraction between the two.
template <typename R>
__device__ __forceinline__ void entropy_vars4(R b, R ux, R uy, R W, R lnr, R lnb, R c1g, R ig, R V[4])
{
    V[0] = c1g + lnr + ig * lnb + b;
    V[1] = b * ux;
    V[2] = b * uy;
    V[3] = -b * W;
}
template <>
__device__ __forceinline__ void entropy_vars4<double>(double b, double ux, double uy, double W, double lnr,
                                                      double lnb, double c1g, double ig, double V[4])
{
    V[0] = __dadd_rn(__fma_rn(ig, lnb, __dadd_rn(c1g, lnr)), b);
    V[1] = __dmul_rn(b, ux);
    V[2] = __dmul_rn(b, uy);
    V[3] = -__dmul_rn(b, W);
}
template <>
__device__ __forceinline__ void entropy_vars4<float>(float b, float ux, float uy, float W, float lnr, float lnb,
                                                     float c1g, float ig, float V[4])
{
    V[0] = __fadd_rn(__fmaf_rn(ig, lnb, __fadd_rn(c1g, lnr)), b);
    V[1] = __fmul_rn(b, ux);
    V[2] = __fmul_rn(b, uy);
    V[3] = -__fmul_rn(b, W);
}

// d = b - a of two nodes' entropy variables, one rounding each (in FP64 and FP32
// never contracted with what forms or uses them)
template <typename R>
__device__ __forceinline__ void v_diff(const R a[4], const R b[4], R d[4])
{
#pragma unroll
    for (int q = 0; q < 4; ++q) d[q] = sub_<R>(b[q], a[q]);
}

// the type of the switch's tolerance: FP32 in both forms
template <typename R> struct TolT { using type = R; };
template <> struct TolT<double> { using type = float; };
__device__ __forceinline__ float to_tol(double x) { return d2f_int(x); }
template <typename R> __device__ __forceinline__ R to_tol(R x) { return x; }

// the six quantities of stencil node k: get(k, j), j = 0..5: beta, u_x, u_y, W, ln rho,
// ln beta
template <typename R, typename GET>
struct NodeStencil {
    GET get;
    __device__ __forceinline__ void state(int k, R &b, R &ux, R &uy) const
    {
        b = get(k, 0);
        ux = get(k, 1);
        uy = get(k, 2);
    }
    __device__ __forceinline__ void V(int k, R c1g, R ig, R v[4]) const
    {
        entropy_vars4<R>(get(k, 0), get(k, 1), get(k, 2), get(k, 3), get(k, 4), get(k, 5), c1g, ig, v);
    }
    __device__ __forceinline__ void dV(int k, R c1g, R ig, R d[4]) const
    {
        R a[4], b[4];
        V(k, c1g, ig, a);
        V(k + 1, c1g, ig, b);
        v_diff<R>(a, b, d);
    }
    __device__ __forceinline__ void V32(int k, R c1g, R ig, typename TolT<R>::type v[4]) const
    {
        R a[4];
        V(k, c1g, ig, a);
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = to_tol(a[q]);
    }
};
// ... read straight from the node arrays
struct QGet {
    const double *q;
    long long P, c0, sd;
    int off;
    __device__ __forceinline__ double operator()(int k, int j) const
    {
        const int f = j == 0 ? Q_BETA : (j == 1 ? Q_UX : (j == 2 ? Q_UY : (j == 3 ? Q_W : (j == 4 ? Q_LNR : Q_LNB))));
        return q[f * P + c0 + (k - off) * sd];
    }
};
// ... from the FP32 copies (the mixed form)
struct QGet32 {
    const float *q;
    long long P, c0, sd;
    int off;
    __device__ __forceinline__ float operator()(int k, int j) const
    {
        const int f = j == 0 ? Q32_B
                    : (j == 1 ? Q32_UX : (j == 2 ? Q32_UY : (j == 3 ? Q32_W : (j == 4 ? Q32_LNR : Q32_LNB))));
        return q[f * P + c0 + (k - off) * sd];
    }
};
// ... from an array (the operation count)
template <typename R>
struct ArrGet {
    const R (*a)[6];
    __device__ __forceinline__ R operator()(int k, int j) const { return a[k][j]; }
};

// jump_sign64 of a jump against its FP64 terms, e the wave's row
template <typename ST>
static __device__ __noinline__ int jump_sign_node64(ST st, int k, double c1g, double ig, double nx, double ny, double e0,
                                                    double e1, double e2, double e3, double jump, double sign_tol)
{
    double scale = 0.0;
#pragma unroll 1
    for (int side = 0; side < 2; ++side) {
        double V[4];
        st.V(k + side, c1g, ig, V);
        scale += fabs(e0 * V[0]) + fabs(e1 * (nx * V[1] + ny * V[2])) + fabs(e2 * (nx * V[2] - ny * V[1])) + fabs(e3 * V[3]);
    }
    return jump_sign64(jump, sign_tol, scale);
}

// The ES dissipation 1/2 lambda^ T^-1 R Y <<V~>> of eq. ESFlux_HO at one
// interface, subtracted from the EC flux F.  nvx, nvy, jt: the interface
// metrics (mean of the two nodes); rho0/1: the density at the two interface nodes
// (log-mean arguments); st: the w + 1 stencil nodes, the interface nodes at
// k = (w-1)/2 and (w+1)/2, with state (beta, u_x, u_y), differences dV(k) = V_{k+1} -
// V_k of the entropy variables, and V32 their FP32 values (for the switch's
// tolerance).  The eigen-system is taken at rho = {{rho}}^ln,
// u = {{u}}, p = {{rho}}/{{beta}}; Y has sign 0 for jumps at rounding level.
// Sums of two products are written as the fused operation, so that the kernels that
// inline this round them alike.
// The dissipation depends on differences of V alone, so they are projected (w of
// them) rather than the w + 1 values.
template <typename R, int WW, typename ST>
__device__ __forceinline__ void es_dissipation(R nvx, R nvy, R jt, const LmV<R> &rho0, const LmV<R> &rho1,
                                               const ST &st, const Phys &ph, R F[4])
{
    constexpr int OFF = (WW - 1) / 2;
    using S = typename TolT<R>::type;
    const R half = (R)0.5, one = (R)1;
    const R gam = (R)ph.gamma;
    R n2 = fma_<R>(nvx, nvx, nvy * nvy);
    R iLk = qrsq<R>(n2);
    R Lk = n2 * iLk;
    R nx = nvx * iLk, ny = nvy * iLk;
    R rho, irho, b0, b1, u0, u1, y0, y1;
    logmean2<R>(rho0, rho1, ph.ln_thr, rho, irho);
    st.state(OFF, b0, u0, y0);
    st.state(OFF + 1, b1, u1, y1);
    R ux = half * (u0 + u1), uy = half * (y0 + y1);
    R p = (rho0.v + rho1.v) * qrcp<R>(b0 + b1);
    R w2 = fma_<R>(uy, uy, fma_<R>(ux, ux, one));
    R iW = qrsq<R>(w2);
    R W = w2 * iW;
    const R ig = (R)ph.gm1i, c1g = gam * ig;
    R E[4][4], lm, lp;
    eigen_rhd<R>(gam, c1g, (R)ph.igg, rho, p, fma_<R>(nx, ux, ny * uy), fma_<R>(nx, uy, -(ny * ux)), W, iW, E, lm,
                 lp);
    R lhat = vmax(fab<R>(fma_<R>(Lk, lm, jt)), fab<R>(fma_<R>(Lk, lp, jt)));
    // |T V| summed over the two interface nodes, for the switch's tolerance
    S aT[4];
    {
        S V0[4], V1[4];
        const S nx_ = to_tol(nx), ny_ = to_tol(ny);
        st.V32(OFF, c1g, ig, V0);
        st.V32(OFF + 1, c1g, ig, V1);
        aT[0] = fab<S>(V0[0]) + fab<S>(V1[0]);
        aT[1] = fab<S>(nx_ * V0[1] + ny_ * V0[2]) + fab<S>(nx_ * V1[1] + ny_ * V1[2]);
        aT[2] = fab<S>(nx_ * V0[2] - ny_ * V0[1]) + fab<S>(nx_ * V1[2] - ny_ * V1[1]);
        aT[3] = fab<S>(V0[3]) + fab<S>(V1[3]);
        if constexpr (std::is_same<S, float>::value) jump_terms<R, 4>(aT);
    }
    // projected differences, the rotation T folded into the projection rows once per
    // interface
    R Dt[WW][4];
    {
        R Ar[4][4];
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            Ar[m][0] = E[m][0];
            Ar[m][1] = fma_<R>(nx, E[m][1], -(ny * E[m][2]));
            Ar[m][2] = fma_<R>(ny, E[m][1], nx * E[m][2]);
            Ar[m][3] = E[m][3];
        }
#pragma unroll
        for (int k = 0; k < WW; ++k) {
            R D[4];
            st.dV(k, c1g, ig, D);
#pragma unroll
            for (int m = 0; m < 4; ++m)
                Dt[k][m] = fma_<R>(Ar[m][3], D[3], fma_<R>(Ar[m][2], D[2], fma_<R>(Ar[m][1], D[1], Ar[m][0] * D[0])));
        }
    }
    R d[4] = {(R)0, (R)0, (R)0, (R)0};
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        R jw;
        if constexpr (WW == 5)
            jw = weno5_jump<R>(Dt[0][m], Dt[1][m], Dt[2][m], Dt[3][m], Dt[4][m], (R)(4.0 * ph.eps));
        else
            jw = weno3_jump<R>(Dt[0][m], Dt[1][m], Dt[2][m], (R)ph.eps);
        const R jump = Dt[OFF][m];
        // a jump within sign_tol of the magnitudes forming V~_m at the two
        // interface nodes is rounding noise: its sign is 0 (so Y = 0)
        const S scale = fab<S>(to_tol(E[m][0])) * aT[0] + fab<S>(to_tol(E[m][1])) * aT[1] +
                        fab<S>(to_tol(E[m][2])) * aT[2] + fab<S>(to_tol(E[m][3])) * aT[3];
        int sj;
        if constexpr (std::is_same<S, float>::value) {
            sj = jump_sign(jump, ph.sign_tol, scale);
            if constexpr (std::is_same<R, double>::value)
                if (sj == JUMP_UNSURE)
                    sj = jump_sign_node64(st, OFF, c1g, ig, nx, ny, E[m][0], E[m][1], E[m][2], E[m][3], jump, ph.sign_tol);
        } else {
            sj = le(fab<S>(jump), (S)ph.sign_tol * scale) ? 0 : sgn_d(jump);
        }
        const R z = (sgn_d(jw) == sj) ? jw : (R)0;
#pragma unroll
        for (int a = 0; a < 4; ++a) d[a] = fma_<R>(E[m][a], z, d[a]);
    }
    R hl = half * lhat;
    F[0] = fma_<R>(-hl, d[0], F[0]);
    F[1] = fma_<R>(-hl, fma_<R>(nx, d[1], -(ny * d[2])), F[1]);
    F[2] = fma_<R>(-hl, fma_<R>(ny, d[1], nx * d[2]), F[2]);
    F[3] = fma_<R>(-hl, d[3], F[3]);
}

// anchors A in [-P, n_dir - 1] along the sweep, every line of the other
// index: the sites of tile t (sweep_site)
template <typename R, int P>
__device__ __forceinline__ void pairs_tile(const ProbArg &pa, const Phys &ph, const double *__restrict__ q,
                                           const float *__restrict__ q32, R *__restrict__ pairs, int dir, int tx,
                                           long long t)
{
    constexpr bool F32 = std::is_same<R, float>::value;
    ProbDesc D;
    long long lb;
    locate_tile(pa, t, D, lb);
    const Geom &g = D.g;
    q += (long long)NQ * D.op;
    if (F32) q32 += (long long)NQ32 * D.op;
    pairs += (long long)2 * PMAX * 4 * D.op;
    int i, j;
    if (!sweep_site(g, dir, P, tx, lb, i, j)) return;
    const long long c0 = pidx(g, i, j);
    const long long sd = dir == 0 ? 1 : g.px;
    // metrics in the working precision: FP64 node arrays or their FP32 copies
    using MT = typename std::conditional<F32, float, double>::type;
    const MT *Mt, *Mx, *My;
    if constexpr (F32) {
        Mt = q32 + (Q32_MT0 + dir) * g.P;
        Mx = q32 + (Q32_M00 + 2 * dir) * g.P;
        My = q32 + (Q32_M01 + 2 * dir) * g.P;
    } else {
        Mt = q + (Q_MT0 + dir) * g.P;
        Mx = q + (Q_M00 + 2 * dir) * g.P;
        My = q + (Q_M01 + 2 * dir) * g.P;
    }
    const R gm1inv = (R)(1.0 / (ph.gamma - 1.0));
    NodeV<R> l = load_node<R>(g, q, q32, c0);
    const MT mtl = Mt[c0], mxl = Mx[c0], myl = My[c0];
#pragma unroll
    for (int n = 1; n <= P; ++n) {
        const long long cr = c0 + n * sd;
        NodeV<R> r = load_node<R>(g, q, q32, cr);
        R mt = (R)((MT)0.5 * (mtl + Mt[cr]));
        R mx = (R)((MT)0.5 * (mxl + Mx[cr]));
        R my = (R)((MT)0.5 * (myl + My[cr]));
        R out[4];
        ec_pair<R>(l, r, mt, mx, my, gm1inv, ph.ln_thr, out);
#pragma unroll
        for (int a = 0; a < 4; ++a)
            pairs[((long long)((dir * PMAX + (n - 1)) * 4 + a)) * g.P + c0] = out[a];
    }
}

// the blocks stride over the ntiles tiles (one tile each when the grid has
// ntiles blocks; a persistent grid when it has fewer)
template <typename R, int P>
__global__ void __launch_bounds__(128) k_pairs(ProbArg pa, Phys ph, const double *__restrict__ q,
                                               const float *__restrict__ q32, R *__restrict__ pairs, int dir, int tx,
                                               long long ntiles)
{
    for (long long t = blockIdx.x; t < ntiles; t += gridDim.x) pairs_tile<R, P>(pa, ph, q, q32, pairs, dir, tx, t);
}

// interfaces between left node L in [-1, n_dir - 1] and L + 1: the sites of
// tile t (sweep_site)
template <typename R, int P, int WW>
__device__ __forceinline__ void iface_tile(const ProbArg &pa, const Phys &ph, const double *__restrict__ q,
                                           const float *__restrict__ q32, const R *__restrict__ pairs,
                                           R *__restrict__ iflux, int dir, int tx, long long t)
{
    constexpr bool F32 = std::is_same<R, float>::value;
    using MT = typename std::conditional<F32, float, double>::type;
    ProbDesc D;
    long long lb;
    locate_tile(pa, t, D, lb);
    const Geom &g = D.g;
    q += (long long)NQ * D.op;
    if (F32) q32 += (long long)NQ32 * D.op;
    pairs += (long long)2 * PMAX * 4 * D.op;
    iflux += (long long)2 * 5 * D.op;
    int i, j;
    if (!sweep_site(g, dir, 1, tx, lb, i, j)) return;
    const long long c0 = pidx(g, i, j);
    const long long sd = dir == 0 ? 1 : g.px;
    // metrics in the working precision: FP64 node arrays or their FP32 copies
    const MT *Mt, *Mx, *My;
    if constexpr (F32) {
        Mt = q32 + (Q32_MT0 + dir) * g.P;
        Mx = q32 + (Q32_M00 + 2 * dir) * g.P;
        My = q32 + (Q32_M01 + 2 * dir) * g.P;
    } else {
        Mt = q + (Q_MT0 + dir) * g.P;
        Mx = q + (Q_M00 + 2 * dir) * g.P;
        My = q + (Q_M01 + 2 * dir) * g.P;
    }

    // eq. ECFlux_O2p: sum_n alpha_{p,n} sum_{s<n} F~(A - s, A - s + n)
    R F[4] = {(R)0, (R)0, (R)0, (R)0};
    MT Ft = (MT)0;
#pragma unroll
    for (int n = 1; n <= P; ++n) {
        R Fs[4] = {(R)0, (R)0, (R)0, (R)0};
        MT Fts = (MT)0;
#pragma unroll
        for (int s = 0; s < n; ++s) {
            const long long ca = c0 - s * sd;
            const R *pr = pairs + ((long long)(dir * PMAX + (n - 1)) * 4) * g.P + ca;
#pragma unroll
            for (int a = 0; a < 4; ++a) Fs[a] += pr[a * g.P];
            Fts += (MT)0.5 * (Mt[ca] + Mt[ca + n * sd]);
        }
        const R an = (R)ph.alpha[n - 1];
#pragma unroll
        for (int a = 0; a < 4; ++a) F[a] = fma_<R>(an, Fs[a], F[a]);
        Ft += (MT)ph.alpha[n - 1] * Fts;
    }

    if constexpr (WW > 0) {
        // eq. ESFlux_HO: subtract 1/2 lambda^ T^-1 R Y <<V~>>
        const long long c1 = c0 + sd;
        const R nvx = (R)((MT)0.5 * (Mx[c0] + Mx[c1])), nvy = (R)((MT)0.5 * (My[c0] + My[c1]));
        const R jt = (R)((MT)0.5 * (Mt[c0] + Mt[c1]));
        if constexpr (F32) {
            const LmV<R> rho0 = lmv_f32(q[Q_RHO * g.P + c0], q32[Q32_R * g.P + c0], q32[Q32_LNR * g.P + c0]);
            const LmV<R> rho1 = lmv_f32(q[Q_RHO * g.P + c1], q32[Q32_R * g.P + c1], q32[Q32_LNR * g.P + c1]);
            NodeStencil<R, QGet32> st{{q32, g.P, c0, sd, (WW - 1) / 2}};
            es_dissipation<R, WW>(nvx, nvy, jt, rho0, rho1, st, ph, F);
        } else {
            const LmV<R> rho0 = {q[Q_RHO * g.P + c0], q[Q_LNR * g.P + c0]};
            const LmV<R> rho1 = {q[Q_RHO * g.P + c1], q[Q_LNR * g.P + c1]};
            NodeStencil<R, QGet> st{{q, g.P, c0, sd, (WW - 1) / 2}};
            es_dissipation<R, WW>(nvx, nvy, jt, rho0, rho1, st, ph, F);
        }
    }
    R *out = iflux + (long long)(dir * 5) * g.P + c0;
#pragma unroll
    for (int a = 0; a < 4; ++a) out[a * g.P] = F[a];
    out[4 * g.P] = (R)Ft;
}

template <typename R, int P, int WW>
__global__ void __launch_bounds__(128) k_iface(ProbArg pa, Phys ph, const double *__restrict__ q,
                                               const float *__restrict__ q32, const R *__restrict__ pairs,
                                               R *__restrict__ iflux, int dir, int tx, long long ntiles)
{
    for (long long t = blockIdx.x; t < ntiles; t += gridDim.x)
        iface_tile<R, P, WW>(pa, ph, q, q32, pairs, iflux, dir, tx, t);
}

inline long long tiles_of(const LaunchDom &L) { return L.ntiles < 0 ? (long long)L.nblk : L.ntiles; }

#if defined(__CUDACC__)
template <typename R, int P>
static void launch_pairs_p(const LaunchDom &L, const Phys &ph, const double *q, const float *q32, R *pairs, int dir,
                           cudaStream_t st)
{
    k_pairs<R, P><<<L.nblk, L.bs, 0, st>>>(L.pa, ph, q, q32, pairs, dir, L.tx, tiles_of(L));
}

template <typename R, int P, int WW>
static void launch_iface_pw(const LaunchDom &L, const Phys &ph, const double *q, const float *q32, const R *pairs,
                            R *iflux, int dir, cudaStream_t st)
{
    k_iface<R, P, WW><<<L.nblk, L.bs, 0, st>>>(L.pa, ph, q, q32, pairs, iflux, dir, L.tx, tiles_of(L));
}

// resident blocks per SM of one instance at block size bs
template <typename K>
static int occ(K kern, int bs)
{
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, bs, 0) != cudaSuccess) n = 1;
    return n > 0 ? n : 1;
}

template <typename R>
int flux_occupancy_t(int kind, int p, int w, int bs)
{
    if (kind == 0) return p == 1 ? occ(k_pairs<R, 1>, bs) : (p == 2 ? occ(k_pairs<R, 2>, bs) : occ(k_pairs<R, 3>, bs));
    auto pick = [&](auto k0, auto k3, auto k5) { return w == 0 ? occ(k0, bs) : (w == 3 ? occ(k3, bs) : occ(k5, bs)); };
    if (p == 1) return pick(k_iface<R, 1, 0>, k_iface<R, 1, 3>, k_iface<R, 1, 5>);
    if (p == 2) return pick(k_iface<R, 2, 0>, k_iface<R, 2, 3>, k_iface<R, 2, 5>);
    return pick(k_iface<R, 3, 0>, k_iface<R, 3, 3>, k_iface<R, 3, 5>);
}

template <typename R>
void launch_pairs_t(const LaunchDom &L, const Phys &ph, const double *q, const float *q32, void *pairs, int dir,
                    cudaStream_t st)
{
    R *pr = (R *)pairs;
    switch (ph.p) {
    case 1: launch_pairs_p<R, 1>(L, ph, q, q32, pr, dir, st); break;
    case 2: launch_pairs_p<R, 2>(L, ph, q, q32, pr, dir, st); break;
    default: launch_pairs_p<R, 3>(L, ph, q, q32, pr, dir, st); break;
    }
}

template <typename R, int P>
static void launch_iface_p(const LaunchDom &L, const Phys &ph, const double *q, const float *q32, const R *pr, R *fl,
                           int dir, cudaStream_t st)
{
    switch (ph.w) {
    case 0: launch_iface_pw<R, P, 0>(L, ph, q, q32, pr, fl, dir, st); break;
    case 3: launch_iface_pw<R, P, 3>(L, ph, q, q32, pr, fl, dir, st); break;
    default: launch_iface_pw<R, P, 5>(L, ph, q, q32, pr, fl, dir, st); break;
    }
}

template <typename R>
void launch_iface_t(const LaunchDom &L, const Phys &ph, const double *q, const float *q32, const void *pairs,
                    void *iflux, int dir, cudaStream_t st)
{
    const R *pr = (const R *)pairs;
    R *fl = (R *)iflux;
    switch (ph.p) {
    case 1: launch_iface_p<R, 1>(L, ph, q, q32, pr, fl, dir, st); break;
    case 2: launch_iface_p<R, 2>(L, ph, q, q32, pr, fl, dir, st); break;
    default: launch_iface_p<R, 3>(L, ph, q, q32, pr, fl, dir, st); break;
    }
}
#endif

}  // namespace esmm

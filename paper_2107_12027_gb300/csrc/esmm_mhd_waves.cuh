// esmm_mhd_waves.cuh -- the waves of the RMHD system along the first axis in
// closed form (included by esmm_mhd.cuh after its arithmetic helpers).
//
// With the 4-velocity u, the comoving field b, e = rho h + b^2 and the covector
// xi = (-lambda, 1, 0, 0), the symmetrized system (entropy variables, with the
// Godunov-Powell term) has the bilinear form
//   X^mu(a, b) = beta { u^mu [S s_a s_b + pi_a pi_b/(Gamma p) + e du_a.du_b +
//                db_a.db_b] + du_a^mu P_b + du_b^mu P_a - b^mu (db_a.du_b + db_b.du_a) },
// s the entropy and pi the pressure perturbation, P = pi + b.db, S = Gamma
// p/(Gamma-1); X^0 is <a, b> = dU(a).dV(b) and X^1 is dV(a).dF~(b).  Its waves
// at xi: with a = u.xi, B = b.xi, k = xi + a u (k.u = 0), k^2 = 1 - lambda^2 + a^2,
//   Alfven:       e a^2 = B^2,   du = s, db = (B/a) s,  s normal to u, k and b;
//   magnetosonic: (e a^2 - B^2)(rho h a^2 - Gamma p k^2) = (rho h - Gamma p)
//                 a^2 k^2 b_t^2,  b_t = b - (B/k^2) k,
// whose du lies in the plane of k and t (t along b_t).  The unknown of the speed
// equations is a (lambda = v_1 - a/W, B = (B_1 + a b^0)/W): slow and Alfven
// speeds close to v_1 then keep their relative accuracy.  Each factor of the
// magnetosonic relation belongs to one wave of a side ("Alfven-like" and
// "sound-like"), and the eigenvector divides by the other factor, so that it
// stays accurate where b_t -> 0 (the vector's error is ~ rounding/|b_t| or less
// and the degenerate pair's span is exact).
//
// Bound: the FP64 pipe.  The same system by a 6 x 6 Gram matrix, Cholesky
// factor and cyclic Jacobi takes ~7,000 FP64 instructions per interface, this
// ~1,000 (a wave ~140); the roots start from FP32 iterations, which cost next to nothing
// beside the FP64 pipe, and take two FP64 Newton steps each.  Measured (GB300,
// 2070 MHz, a perturbed rotor whose speeds are distinct): the 512^2 FP64 step went
// from 51.8 to 20.5 ms, the mixed one from 5.1 to 3.1 ms, a 64^3 blast step from
// 88.3 to 33.2 ms.  Against extended precision the vectors are ~4 times closer in
// the median than the Gram form's (2.2e-15 against 8.0e-15 of a column in FP64),
// 40 times in FP32's worst percent.
#pragma once

namespace esmm {

template <typename R> __device__ __forceinline__ R of_f32(float x);
template <> __device__ __forceinline__ double of_f32<double>(float x) { return f2d_int(x); }
template <> __device__ __forceinline__ float of_f32<float>(float x) { return x; }

// the state of the waves: 4-vectors (index 0 the time component)
template <typename R>
struct MhdBase {
    R W, iW, v1, u[4], b[4], b2, rh, e, gp, beta, ip, rho, B1;
};

// ... from the spatial 4-velocity us and W
template <typename R>
__device__ __forceinline__ void mhd_base_u(R gam, R gg, R rho, R p, R ip, R W, R iW, const R us[3], const R B[3],
                                           MhdBase<R> &s)
{
    s.W = W;
    s.iW = iW;
    s.v1 = us[0] * iW;
    s.rho = rho;
    s.B1 = B[0];
    s.u[0] = W;
    s.b[0] = us[0] * B[0] + us[1] * B[1] + us[2] * B[2];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        s.u[1 + k] = us[k];
        s.b[1 + k] = (B[k] + s.b[0] * us[k]) * iW;
    }
    s.b2 = (B[0] * B[0] + B[1] * B[1] + B[2] * B[2] + s.b[0] * s.b[0]) * (iW * iW);
    s.gp = gam * p;
    s.rh = rho + gg * p;
    s.e = s.rh + s.b2;
    s.ip = ip;
    s.beta = rho * ip;
}

// ... from the primitives w (rotated frame)
template <typename R>
__device__ __forceinline__ void mhd_base(R gam, R gg, const R w[8], MhdBase<R> &s)
{
    const R iW2 = (R)1 - (w[1] * w[1] + w[2] * w[2] + w[3] * w[3]), W = rsq<R>(iW2);
    const R us[3] = {W * w[1], W * w[2], W * w[3]};
    mhd_base_u<R>(gam, gg, w[0], w[4], rcp<R>(w[4]), W, iW2 * W, us, w + 5, s);
    s.v1 = w[1];
}

// the closed form holds (its FP32 root estimates stay in range)
template <typename R>
__device__ __forceinline__ bool mhd_in_range(const MhdBase<R> &s)
{
    const float lim = sizeof(R) == 4 ? 1.0e-12f : 1.0e-25f;
    return to_f32(s.gp) > lim && to_f32(s.e) < 1.0f / lim;
}

// two waves of one cluster: their speeds closer than MHD_CLUSTER_TOL
template <typename R>
__device__ __forceinline__ bool mhd_close(R lam0, R lam1)
{
    return to_f32(lam1 - lam0) < (float)MHD_CLUSTER_TOL;
}

// f(t) of the magnetosonic speeds on the side sg = +-1 (a = sg t, t >= 0),
//   f = cA t^4 - cB t^2 G + h^2 G,  h = c1 + sg t c0,  G = 1 - lambda^2,
// and its derivative; f >= 0 at t = 0, f <= 0 at the Alfven speed, f > 0 at the
// light speed: the slow and the fast speed are its roots on the two sides of
// the Alfven speed.
template <typename R>
__device__ __forceinline__ void mhd_quartic(R cA, R cB, R c1, R c0s, R v1, R iWs, R t, R &f, R &df)
{
    // c0s = sg c0, iWs = sg / W
    const R lam = v1 - t * iWs, G = ((R)1 - lam) * ((R)1 + lam), dG = (R)2 * lam * iWs;
    const R h = c1 + t * c0s, t2 = t * t, q = h * h - cB * t2;
    f = cA * t2 * t2 + q * G;
    df = (R)4 * cA * t2 * t + (R)2 * (h * c0s - cB * t) * G + q * dG;
}

// FP32 estimates of the slow and fast roots of one side (all coefficients
// divided by rho h), bracketed Newton
__device__ __forceinline__ void mhd_roots32(float cA, float cB, float c1, float c0s, float v1, float iWs, float tA,
                                            float tmax, float &tslow, float &tfast, bool want_slow)
{
    float t = tmax;
#pragma unroll 1
    for (int it = 0; it < 24; ++it) {   // from the right end: monotone
        float f, df;
        mhd_quartic<float>(cA, cB, c1, c0s, v1, iWs, t, f, df);
        if (!(df > 0.0f)) break;
        const float tn = fmaxf(t - f * __frcp_rn(df), tA);
        const bool done = fabsf(tn - t) <= 1.0e-6f * t;
        t = tn;
        if (done) break;
    }
    tfast = t;
    if (!want_slow) return;
    // without the t^4 term the root is linear; it is a lower bound
    const float t0 = fabsf(c1) * __frcp_rn(sqrtf(cB) - (c1 < 0.0f ? -c0s : c0s));
    float lo = fminf(t0, tA), hi = tA;
    t = lo;
    if (t > 1.0e-12f)   // (below, the t^4 term is far under rounding)
#pragma unroll 1
        for (int it = 0; it < 24; ++it) {
            float f, df;
            mhd_quartic<float>(cA, cB, c1, c0s, v1, iWs, t, f, df);
            if (f > 0.0f) lo = t; else hi = t;
            float tn = t - f * __frcp_rn(df);
            if (!(tn >= lo && tn <= hi)) tn = 0.5f * (lo + hi);
            const bool done = fabsf(tn - t) <= 1.0e-6f * t;
            t = tn;
            if (done) break;
        }
    tslow = t;
}

template <typename R> __device__ __forceinline__ bool is_neg(R x) { return x < (R)0; }
template <typename R> __device__ __forceinline__ bool is_zero(R x) { return x == (R)0; }
template <> __device__ __forceinline__ bool is_neg<double>(double x) { return (conv_bits64(x) >> 63) != 0; }
template <> __device__ __forceinline__ bool is_zero<double>(double x) { return (conv_bits64(x) << 1) == 0; }

__device__ __forceinline__ bool positive_finite(float x) { return x > 0.0f && x < __FLT_MAX__; }
__device__ __forceinline__ bool positive_finite(double x) { return conv_bits64(x) - 1ull < 0x7fefffffffffffffull; }

// the smaller and larger of two numbers, b >= 0: in FP64 by their bits (non-negative
// numbers order like them and a negative one lies below; FP64 compares cost FP64-pipe slots)
__device__ __forceinline__ float lesser_nn(float a, float b) { return fminf(a, b); }
__device__ __forceinline__ float larger_nn(float a, float b) { return fmaxf(a, b); }
__device__ __forceinline__ double lesser_nn(double a, double b)
{
    return (long long)conv_bits64(a) < (long long)conv_bits64(b) ? a : b;
}
__device__ __forceinline__ double larger_nn(double a, double b)
{
    return (long long)conv_bits64(a) > (long long)conv_bits64(b) ? a : b;
}

// Newton in R from the FP32 estimate t, kept in [lo, hi] (0 <= lo).  The step divides
// through an FP32 reciprocal (a relative slope error contracts the error by
// that much per step); a step below 1e-9 t leaves an error under rounding.
template <typename R>
__device__ __forceinline__ R mhd_polish(R cA, R cB, R c1, R c0s, R v1, R iWs, R t, R lo, R hi)
{
    const int most = sizeof(R) == 4 ? 2 : 12;
#pragma unroll 1
    for (int it = 0; it < most; ++it) {
        R f, df;
        mhd_quartic<R>(cA, cB, c1, c0s, v1, iWs, t, f, df);
        const R dt = f * of_f32<R>(__frcp_rn(to_f32(df)));
        const float d32 = fabsf(to_f32(dt));
        const bool done = !(d32 > (sizeof(R) == 4 ? 1.0e-4f : 1.0e-9f) * to_f32(t));
        if (d32 == d32) t = larger_nn(lesser_nn(t - dt, hi), lo);   // (a NaN step, f = f' = 0, ends the loop)
        if (done) break;
    }
    return t;
}

template <typename R>
__device__ __forceinline__ R mdot(const R a[4], const R b[4])
{
    return a[1] * b[1] + a[2] * b[2] + a[3] * b[3] - a[0] * b[0];
}

// the 4-vector normal to u, xi = (lambda, 1, 0, 0) and c
template <typename R>
__device__ __forceinline__ void mcross(const R u[4], R lam, const R c[4], R o[4])
{
    const R q = u[2] * c[3] - u[3] * c[2], A = u[0] - lam * u[1], C = c[0] - lam * c[1];
    o[0] = q;
    o[1] = lam * q;
    o[2] = c[3] * A - u[3] * C;
    o[3] = u[2] * C - c[2] * A;
}

// The two roots of a side where the Alfven and the sound speed nearly coincide
// (with b_t -> 0 a double root of f): with tS the root of the sound factor
//   f = (t - tA)(t - tS) H(t) - C(t),  H > 0,  C = (rho h - Gamma p) t^2 |k x b|^2,
// so t = m +- sqrt((tA - tS)^2/4 + C/H), m their mean, a contraction by ~|b_t| per
// step and well conditioned at the double root.
template <typename R>
__device__ __noinline__ void mhd_near_triple(const MhdBase<R> &s, R sqe, R sg, R tA, bool want_slow, R &ts, R &tf)
{
    const R sgm = s.B1 < (R)0 ? -(R)1 : (R)1;
    const R S2 = s.rh - s.gp + s.gp * s.iW * s.iW, hb = s.gp * s.v1 * sg * s.iW;
    const R q = sq_rt<R>(hb * hb + S2 * s.gp * ((R)1 - s.v1 * s.v1)), iS2 = rcp<R>(S2);
    const R tS = (hb + q) * iS2, tS2 = (q - hb) * iS2;   // roots tS and -tS2
    const R dA = sqe - sgm * sg * s.b[0] * s.iW;
    const R m = (R)0.5 * (tA + tS), hd = (R)0.5 * (tA - tS);
    for (int r = 0; r < (want_slow ? 2 : 1); ++r) {
        R t = r == 0 ? tf : ts;
#pragma unroll 1
        for (int it = 0; it < 40; ++it) {
            const R a = sg * t, lam = s.v1 - a * s.iW;
            R sv[4];
            mcross<R>(s.u, lam, s.b, sv);
            const R H = dA * (sqe * t + sgm * (s.B1 + a * s.b[0]) * s.iW) * S2 * (t + tS2);
            const R w = sq_rt<R>(hd * hd + (s.rh - s.gp) * t * t * mdot<R>(sv, sv) * rcp<R>(H));
            const R tn = r == 0 ? m + w : m - w;
            const bool done = !(fab<R>(tn - t) > (sizeof(R) == 4 ? (R)1.0e-7 : (R)2.0e-16) * tn);
            t = tn;
            if (done) break;
        }
        (r == 0 ? tf : ts) = t;
    }
}

// coefficients of both sides
template <typename R>
struct MhdCoef {
    R sqe, cA, cB, c1, c0, We;
};
template <typename R>
__device__ __forceinline__ void mhd_coef(const MhdBase<R> &s, MhdCoef<R> &k)
{
    const R q = s.rh * qrcp<R>(s.gp);
    k.sqe = s.e * qrsq<R>(s.e);
    k.cA = s.rh * (q - (R)1);
    k.cB = s.rh + s.b2 * q;
    k.c1 = s.B1 * s.iW;
    k.c0 = s.b[0] * s.iW;
    k.We = s.W * k.sqe;
}

// the Alfven and magnetosonic |a| of the side sg
template <typename R>
__device__ __forceinline__ void mhd_side(const MhdBase<R> &s, const MhdCoef<R> &kc, int sg, bool want_slow, R &tA, R &tslow,
                                         R &tfast)
{
    const R sgr = (R)sg, sqe = kc.sqe, cA = kc.cA, cB = kc.cB, c1 = kc.c1;
    const R c0s = sgr * kc.c0, iWs = sgr * s.iW;
    const R tmax = s.W * ((R)1 + sgr * s.v1);
    const bool neg = is_neg(s.B1);
    tA = fab<R>(s.B1) * qrcp<R>(kc.We - (neg ? -sgr : sgr) * s.b[0]);
    if (to_f32(tA) < (sizeof(R) == 4 ? 1.0e-18f : 1.0e-30f)) tA = (R)0;   // (the speed v_1 at rounding)
    float fs = 0.0f, ff;
    const float irh = __frcp_rn(to_f32(s.rh)), qrh = sqrtf(irh);
    mhd_roots32(to_f32(cA) * irh, to_f32(cB) * irh, to_f32(c1) * qrh, to_f32(c0s) * qrh, to_f32(s.v1), to_f32(iWs),
                to_f32(tA), to_f32(tmax), fs, ff, want_slow);
    // (the sound speed and the fast speed within 2% of the Alfven speed)
    bool near;
    {
        const float gp = to_f32(s.gp) * irh, S2 = 1.0f - gp + gp * to_f32(s.iW) * to_f32(s.iW);
        const float v1 = to_f32(s.v1), iW = to_f32(iWs), fA = to_f32(tA), hb = gp * v1 * iW;
        const float tS = (hb + sqrtf(hb * hb + S2 * gp * (1.0f - v1 * v1))) * __frcp_rn(S2);
        near = fabsf(tS - fA) <= 0.02f * fA && ff - fA <= 0.02f * fA;
    }
    tfast = of_f32<R>(ff);
    if (!near) tfast = mhd_polish<R>(cA, cB, c1, c0s, s.v1, iWs, tfast, tA, tmax);
    tslow = (R)0;
    if (want_slow && !is_zero(tA)) {
        if (fs > 1.0e-12f) {
            tslow = mhd_polish<R>(cA, cB, c1, c0s, s.v1, iWs, of_f32<R>(fs), (R)0, tA);
        } else {   // an FP32 estimate that underflowed: the linear root in R
            tslow = lesser_nn(fab<R>(c1) * rcp<R>(sq_rt<R>(cB) - (neg ? -c0s : c0s)), tA);
        }
    }
    if (near) mhd_near_triple<R>(s, sqe, sgr, tA, want_slow, tslow, tfast);
}

// One wave: perturbations (d rho, du, db, dp), scaled to <., .> = 1
template <typename R>
struct MhdWave {
    R rho, p, u[4], b[4];
};

// dU of a wave: (D, m, E, B)
template <typename R>
__device__ __forceinline__ void mhd_wave_dU(const MhdBase<R> &s, R gg, const MhdWave<R> &q, R dU[8])
{
    const R bdb = mdot<R>(s.b, q.b);
    const R de = q.rho + gg * q.p + (R)2 * bdb;
    const R c0 = de * s.W + s.e * q.u[0], c1 = s.e * s.W;
    dU[0] = s.rho * q.u[0] + s.W * q.rho;
#pragma unroll
    for (int k = 1; k < 4; ++k) dU[k] = c0 * s.u[k] + c1 * q.u[k] - q.b[0] * s.b[k] - s.b[0] * q.b[k];
    dU[4] = de * s.W * s.W + (R)2 * (c1 * q.u[0] - s.b[0] * q.b[0]) - (q.p + bdb);
#pragma unroll
    for (int k = 1; k < 4; ++k) dU[4 + k] = q.u[0] * s.b[k] + s.W * q.b[k] - q.u[k] * s.b[0] - s.u[k] * q.b[0];
}

// One of the four waves of speed v_1 at B_1 = 0, spanned by du or db along s or t
// with P = 0; du.db = 0, and m du^2 is e du^2 - (b.du)^2: m = e along s, rho h along t
template <typename R>
__device__ __forceinline__ void mhd_still_wave(const MhdBase<R> &s, bool along_u, R m, const R d[4], MhdWave<R> &q)
{
    const R bd = mdot<R>(s.b, d);
    q.p = along_u ? (R)0 : -bd;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        q.u[i] = along_u ? d[i] : (R)0;
        q.b[i] = along_u ? bd * s.u[i] : d[i];   // (db = (b.du) u)
    }
    const R d2 = mdot<R>(d, d);
    const R n2 = s.beta * s.W * (along_u ? m * d2 : d2 + bd * bd * rcp<R>(s.gp));
    const R sc = rsq<R>(n2);
    q.p *= sc;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        q.u[m] *= sc;
        q.b[m] *= sc;
    }
    q.rho = q.p * s.rho * rcp<R>(s.gp);   // adiabatic
}

// The wave of kind 0 (fast), 1 (Alfven), 2 (slow) on the side sg, given its |a| = t; c
// spans with u and xi the wave's plane (b's direction, of size 1 so that s^2 and t^2 are
// normal numbers under any field, or a coordinate axis where b lies along k).
// With k^2 = 1 - lambda^2 + a^2, s normal to u, xi and c, t normal to u, xi and s
// (t^2 = s^2 k^2), every wave has
//   du = y = y_t t + y_k k (Alfven: s),  d p = Gamma p pk,  d rho = rho pk,
//   db = r y + pk b + (b.y) u,  r = B/a,
// so that the norm and dU take scalars instead of 4-vector products, and one code path for the
// two magnetosonic forms, which differ between the lanes of a warp.  The norm is
//   X^0(q, q) = beta { E W (1 - v_1 lambda)/k^2 + 2 t^0 y_t dp },
//   E = dp pk + rho h y^2 + z^2 t^2 (1 + a^2/k^2),  z = r y_t + pk (b.t)/t^2,  t^2 = s^2 k^2
// (the parts of X^mu along k follow from xi.X = 0 and along t all but one cancel; the Alfven
// waves': 2 beta y^2 (W e - b^0 r)): E is a sum of squares, where the energy's own terms
// W (e y^2 + db^2) + 2 (y^0 P - b^0 db.y) cancel to 1/W^2 of their size under strong fields
// (FP32 norms at W = 10 .. 20, b^2 > rho h were off by 8% in the median, 6% of them negative; now
// 6e-4).  out: dU, and the du (4-vector) and dp it belongs to; FULL: the perturbations q
// instead of dU; false where rounding leaves no positive norm (FP32 above W ~ 200).
template <typename R, bool FULL>
__device__ __forceinline__ bool mhd_wave(const MhdBase<R> &s, R sqe, R gg, int kind, int sg, R tw, bool alf_like,
                                         const R c[4], MhdWave<R> &q, R dU[8])
{
    const R a = (R)sg * tw, lam = s.v1 - a * s.iW;
    R sv[4], tv[4];
    mcross<R>(s.u, lam, c, sv);
    mcross<R>(s.u, lam, sv, tv);
    if (kind != 0 && is_zero(tw)) {
        mhd_still_wave<R>(s, sg > 0, kind == 1 ? s.e : s.rh, kind == 1 ? sv : tv, q);
        if constexpr (!FULL) mhd_wave_dU<R>(s, gg, q, dU);
        return true;
    }
    R y[4], by, r, pk, n2;
    if (kind == 1) {
        R s2[4];
        mcross<R>(s.u, lam, tv, s2);   // (normal to u and xi at rounding)
#pragma unroll
        for (int m = 0; m < 4; ++m) y[m] = s2[m];
        r = is_neg(s.B1) ? (R)-sg * sqe : (R)sg * sqe;
        pk = (R)0;
        by = mdot<R>(s.b, y);
        n2 = (R)2 * mdot<R>(y, y) * (s.W * s.e - s.b[0] * r);
    } else {
        const R a2 = a * a, k2 = ((R)1 - lam) * ((R)1 + lam) + a2, Bx = (s.B1 + a * s.b[0]) * s.iW;
        const R bt = mdot<R>(s.b, tv), s2 = mdot<R>(sv, sv), ra2 = s.rh * a2, gk2 = s.gp * k2;
        r = Bx * qrcp<R>(a);
        // alf_like: y = r t - (rho h a (b.t)/Sf) k; else y = a (B (rho h - Gamma p) (b.t)/(rho h
        // De s^2) t - k); one reciprocal for 1/k^2, 1/s^2 and the wave's own quotient
        const bool none = is_zero(bt);
        const R den = none ? (R)1 : (alf_like ? ra2 - gk2 : s.rh * (s.e * a2 - Bx * Bx));
        const R iq = qrcp<R>(k2 * s2 * den), qd = iq * den, ik2 = s2 * qd, is2 = k2 * qd;
        const R cf = (alf_like ? s.rh * s2 : Bx * (s.rh - s.gp)) * (bt * (k2 * iq));
        const R yt = alf_like ? r : a * cf, h = alf_like ? cf : (R)1, yk = -h * a;
        pk = h * k2;
        const R ka = yk * a;   // k = xi + a u
        y[0] = yt * tv[0] + (yk * lam + ka * s.u[0]);
        y[1] = yt * tv[1] + (yk + ka * s.u[1]);
        y[2] = yt * tv[2] + ka * s.u[2];
        y[3] = yt * tv[3] + ka * s.u[3];
        by = yt * bt + yk * Bx;
        const R z = r * yt + h * bt * is2;
        n2 = (h * h * (ra2 + gk2) + s2 * (s.rh * yt * yt + z * z * ((R)1 + a2 * ik2))) * (s.W * ((R)1 - s.v1 * lam)) +
             (R)2 * tv[0] * (yt * (h * gk2));
    }
    R bz = r * by + pk * s.b2;
    const R sc = qrsq<R>(s.beta * n2);
#pragma unroll
    for (int m = 0; m < 4; ++m) y[m] *= sc;
    pk *= sc;
    by *= sc;
    bz *= sc;
    const R p = s.gp * pk;
    const R db0 = r * y[0] + (pk * s.b[0] + by * s.W);
#pragma unroll
    for (int m = 0; m < 4; ++m) q.u[m] = y[m];
    q.p = p;
    q.rho = s.rho * pk;
    if constexpr (FULL) {
        q.b[0] = db0;
#pragma unroll
        for (int k = 1; k < 4; ++k) q.b[k] = r * y[k] + (pk * s.b[k] + by * s.u[k]);
    } else {
        const R c1 = s.e * s.W, de = (s.rho + gg * s.gp) * pk + (R)2 * bz, c0 = de * s.W + s.e * y[0];
        const R hb = y[0] + s.W * pk, hy = s.W * r - s.b[0], hu = s.W * by - db0;
        const R gu = c0 - s.b[0] * by, gy = c1 - s.b[0] * r, gb = db0 + s.b[0] * pk;
        dU[0] = s.rho * hb;
#pragma unroll
        for (int k = 1; k < 4; ++k) {
            dU[k] = gu * s.u[k] + (gy * y[k] - gb * s.b[k]);
            dU[4 + k] = hb * s.b[k] + (hy * y[k] + hu * s.u[k]);
        }
        dU[4] = de * (s.W * s.W) + (R)2 * (c1 * y[0] - s.b[0] * db0) - (p + bz);
    }
    return positive_finite(n2);
}

// The power of two that brings the largest |b_i| into [1, 2); 0 where all are zero or
// subnormal.  (By their bits, off the FP64 pipe.)
template <typename R> __device__ __forceinline__ R inv_binade(const R b[3]);
template <> __device__ __forceinline__ double inv_binade<double>(const double b[3])
{
    uint32_t e = 0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const uint32_t h = (uint32_t)(conv_bits64(b[k]) >> 32) & 0x7fffffffu;
        e = h > e ? h : e;
    }
    e >>= 20;
    return e == 0 ? 0.0 : conv_double((uint64_t)(2046u - e) << 52);
}
template <> __device__ __forceinline__ float inv_binade<float>(const float b[3])
{
    uint32_t e = 0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const uint32_t h = conv_bits32(b[k]) & 0x7fffffffu;
        e = h > e ? h : e;
    }
    e >>= 23;
    return e == 0 ? 0.0f : conv_float((254u - e) << 23);
}

// The six waves' |a| and the frame data shared by their vectors.
template <typename R>
struct MhdSix {
    R t[6], sqe;
    R c[4];          // b by a power of two, of size 1 (0 where there is no field)
    bool alf[2];     // per side: the fast wave is the Alfven-like one
    bool axis[2];    // b along k (|b_t| at rounding level) or no field: c a coordinate axis
};

template <typename R>
__device__ __forceinline__ void mhd_six(const MhdBase<R> &s, MhdSix<R> &x, R lam[6])
{
    MhdCoef<R> kc;
    mhd_coef<R>(s, kc);
    x.sqe = kc.sqe;
    const R cs = inv_binade<R>(s.b + 1);
#pragma unroll
    for (int m = 0; m < 4; ++m) x.c[m] = s.b[m] * cs;
    const float irh = __frcp_rn(to_f32(s.rh)), gp = to_f32(s.gp) * irh;
#pragma unroll
    for (int side = 0; side < 2; ++side) {
        const int sg = side == 0 ? 1 : -1;
        R tA, ts, tf;
        mhd_side<R>(s, kc, sg, true, tA, ts, tf);
        const int o = side == 0 ? 0 : 5, d = side == 0 ? 1 : -1;
        x.t[o] = tf;
        x.t[o + d] = tA;
        x.t[o + 2 * d] = ts;
        // (at equality of the two factors either choice holds)
        const float af = to_f32(tA), lf = to_f32(s.v1) - (float)sg * af * to_f32(s.iW);
        x.alf[side] = af * af > gp * ((1.0f - lf) * (1.0f + lf) + af * af);
        const R la = s.v1 - (R)sg * tA * s.iW;
        R sv[4];
        mcross<R>(s.u, la, x.c, sv);
        const R A = s.u[0] - la * s.u[1], q = (R)(sizeof(R) == 4 ? 1.0e-10 : 1.0e-22) * mdot<R>(x.c, x.c) * A * A;
        x.axis[side] = !(sgn_d(mdot<R>(sv, sv) - q) > 0);
    }
#pragma unroll
    for (int m = 0; m < 6; ++m) lam[m] = m < 3 ? s.v1 - x.t[m] * s.iW : s.v1 + x.t[m] * s.iW;
}

template <typename R, bool FULL>
__device__ __forceinline__ bool mhd_six_wave(const MhdBase<R> &s, const MhdSix<R> &x, R gg, int m, MhdWave<R> &q, R dU[8])
{
    const int side = m < 3 ? 0 : 1, kind = m < 3 ? m : 5 - m;   // 0 fast, 1 Alfven, 2 slow
    const bool alf = side == 0 ? x.alf[0] : x.alf[1], axis = side == 0 ? x.axis[0] : x.axis[1];
    const R c[4] = {axis ? (R)0 : x.c[0], axis ? (R)0 : x.c[1], axis ? (R)1 : x.c[2], axis ? (R)0 : x.c[3]};
    return mhd_wave<R, FULL>(s, x.sqe, gg, kind, side == 0 ? 1 : -1, x.t[m], kind == 0 ? alf : !alf, c, q, dU);
}

// The entropy wave (d rho = 1; its dU[5..7] = 0) and the divergence wave dB = e_1 -
// v_1 v, both of speed v_1.
template <typename R>
__device__ __forceinline__ void mhd_entropy_dU(const MhdBase<R> &s, R igg, R dU[8])
{
    const R q = s.W * s.rho * igg, sr = q * qrsq<R>(q);   // W sqrt(rho/(Gamma/(Gamma-1) W))
    dU[0] = sr;
#pragma unroll
    for (int k = 1; k < 4; ++k) dU[k] = s.u[k] * sr;
    dU[4] = s.W * sr;
#pragma unroll
    for (int k = 5; k < 8; ++k) dU[k] = (R)0;
}
template <typename R>
__device__ __forceinline__ void mhd_divergence_dU(const MhdBase<R> &s, R dU[8])
{
    // db = (v_1/W, dB/W + (v_1/W) v) = e_1/W + (v_1/W)(1, 0): du = dp = 0
    const R b0 = s.v1 * s.iW, b1 = s.iW;
    const R sd = qrsq<R>(s.beta * s.iW * ((R)1 - s.v1 * s.v1));
    const R db0 = b0 * sd, db1 = b1 * sd, bdb = s.b[1] * db1 - s.b[0] * db0, de = (R)2 * bdb, c0 = de * s.W;
    dU[0] = (R)0;
    dU[1] = c0 * s.u[1] - db0 * s.b[1] - s.b[0] * db1;
    dU[2] = c0 * s.u[2] - db0 * s.b[2];
    dU[3] = c0 * s.u[3] - db0 * s.b[3];
    dU[4] = c0 * s.W - (R)2 * (s.b[0] * db0) - bdb;
    dU[5] = s.W * db1 - s.u[1] * db0;
    dU[6] = -s.u[2] * db0;
    dU[7] = -s.u[3] * db0;
}

}  // namespace esmm

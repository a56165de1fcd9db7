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
// ~1,000; the roots start from FP32 iterations, which cost next to nothing
// beside the FP64 pipe, and take two FP64 Newton steps each.  Measured (GB300,
// 2070 MHz, a perturbed rotor whose speeds are distinct): the 512^2 FP64 step went
// from 51.8 to 20.5 ms, the mixed one from 5.1 to 3.1 ms, a 64^3 blast step from
// 88.3 to 33.2 ms.  Against extended precision the vectors are ~8 times closer in
// the median than the Gram form's (1.2e-15 against 8.0e-15 of a column in FP64),
// 50 times in FP32's worst percent.
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

template <typename R>
__device__ __forceinline__ void mhd_base(R gam, R gg, const R w[8], MhdBase<R> &s)
{
    const R iW2 = (R)1 - (w[1] * w[1] + w[2] * w[2] + w[3] * w[3]);
    s.W = rsq<R>(iW2);
    s.iW = iW2 * s.W;
    s.v1 = w[1];
    s.rho = w[0];
    s.B1 = w[5];
    s.u[0] = s.W;
    s.u[1] = s.W * w[1];
    s.u[2] = s.W * w[2];
    s.u[3] = s.W * w[3];
    s.b[0] = s.u[1] * w[5] + s.u[2] * w[6] + s.u[3] * w[7];
#pragma unroll
    for (int k = 0; k < 3; ++k) s.b[1 + k] = (w[5 + k] + s.b[0] * s.u[1 + k]) * s.iW;
    s.b2 = (w[5] * w[5] + w[6] * w[6] + w[7] * w[7] + s.b[0] * s.b[0]) * iW2;
    s.gp = gam * w[4];
    s.rh = w[0] + gg * w[4];
    s.e = s.rh + s.b2;
    s.ip = rcp<R>(w[4]);
    s.beta = w[0] * s.ip;
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

// Newton in R from the FP32 estimate t, kept in [lo, hi].  The step divides
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
        R tn = t - dt;
        tn = tn < lo ? lo : (tn > hi ? hi : tn);   // (a NaN step, f = f' = 0, ends the loop below)
        if (!(fab<R>(dt) > (sizeof(R) == 4 ? (R)1.0e-4 : (R)1.0e-9) * t)) {
            if (dt == dt) t = tn;
            break;
        }
        t = tn;
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

// the Alfven and magnetosonic |a| of the side sg
template <typename R>
__device__ __forceinline__ void mhd_side(const MhdBase<R> &s, R sqe, int sg, bool want_slow, R &tA, R &tslow, R &tfast)
{
    const R sgr = (R)sg;
    const R c0s = sgr * s.b[0] * s.iW, iWs = sgr * s.iW, c1 = s.B1 * s.iW;
    const R igp = rcp<R>(s.gp);
    const R cB = s.rh + s.rh * s.b2 * igp, cA = s.rh * (s.rh * igp - (R)1);
    const R tmax = s.W * ((R)1 + sgr * s.v1);
    tA = fab<R>(s.B1) * rcp<R>(s.W * sqe - (s.B1 < (R)0 ? -sgr : sgr) * s.b[0]);
    if (tA < (R)(sizeof(R) == 4 ? 1.0e-18 : 1.0e-100)) tA = (R)0;
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
    if (want_slow && tA > (R)0) {
        // an FP32 estimate that underflowed: the linear root in R
        R t0 = of_f32<R>(fs);
        if (!(fs > 1.0e-12f))
            t0 = fab<R>(c1) * rcp<R>(sq_rt<R>(cB) - (s.B1 < (R)0 ? -c0s : c0s));
        tslow = fs > 1.0e-12f ? mhd_polish<R>(cA, cB, c1, c0s, s.v1, iWs, t0, (R)0, tA) : (t0 < tA ? t0 : tA);
    }
    if (near) mhd_near_triple<R>(s, sqe, sgr, tA, want_slow, tslow, tfast);
}

// One wave: perturbations (d rho, du, db, dp), scaled to <., .> = 1 by mhd_scale
template <typename R>
struct MhdWave {
    R rho, p, u[4], b[4];
};

// scale to unit X^0 (s = 0 or du = 0 waves: the general form with the entropy part S2 given)
template <typename R>
__device__ __forceinline__ void mhd_scale(const MhdBase<R> &s, MhdWave<R> &q)
{
    const R P = q.p + mdot<R>(s.b, q.b);
    const R n2 = s.beta * (s.W * (q.p * q.p * rcp<R>(s.gp) + s.e * mdot<R>(q.u, q.u) + mdot<R>(q.b, q.b)) +
                           (R)2 * (q.u[0] * P - s.b[0] * mdot<R>(q.b, q.u)));
    const R sc = rsq<R>(n2);
    q.p *= sc;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        q.u[m] *= sc;
        q.b[m] *= sc;
    }
    q.rho = q.p * s.rho * rcp<R>(s.gp);   // adiabatic
}

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

// The wave m = 0 .. 5 of the six (fast, Alfven, slow with a > 0; slow, Alfven,
// fast with a < 0: ascending speeds), given its |a| = t, and the flag of a
// field along k (t then taken along a coordinate axis).
template <typename R>
__device__ __forceinline__ void mhd_wave(const MhdBase<R> &s, R sqe, int kind, int sg, R t, bool alf_like, const R c[4],
                                         MhdWave<R> &q)
{
    const R a = (R)sg * t, lam = s.v1 - a * s.iW;
    R sv[4], tv[4];
    mcross<R>(s.u, lam, c, sv);
    mcross<R>(s.u, lam, sv, tv);
    if (kind != 0 && !(t > (R)0)) {
        // B_1 = 0: the four waves of speed v_1, spanned by du or db along s or t with P = 0
        const R ps = sg > 0 ? (R)0 : -mdot<R>(s.b, kind == 1 ? sv : tv);
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const R d = kind == 1 ? sv[m] : tv[m];
            q.u[m] = sg > 0 ? d : (R)0;
            q.b[m] = sg > 0 ? (R)0 : d;
        }
        q.p = ps;
        if (sg > 0) {   // db = (b.du) u
            const R bd = mdot<R>(s.b, q.u);
#pragma unroll
            for (int m = 0; m < 4; ++m) q.b[m] = bd * s.u[m];
        }
        mhd_scale<R>(s, q);
        return;
    }
    const R r0 = (s.B1 < (R)0 ? -(R)sg : (R)sg);   // the sign of B / a
    if (kind == 1) {   // Alfven: du = s, db = (B/a) s + (b.s) u with b.s = 0
        mcross<R>(s.u, lam, tv, sv);
        const R r = r0 * sqe;
        q.p = (R)0;
        const R bs = mdot<R>(s.b, sv);
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            q.u[m] = sv[m];
            q.b[m] = r * sv[m] + bs * s.u[m];
        }
        mhd_scale<R>(s, q);
        return;
    }
    const R k2 = ((R)1 - lam) * ((R)1 + lam) + a * a;
    const R Bx = (s.B1 + a * s.b[0]) * s.iW;
    R kv[4] = {lam + a * s.u[0], (R)1 + a * s.u[1], a * s.u[2], a * s.u[3]};
    const R bt = mdot<R>(s.b, tv);
    R y[4], z[4];
    if (alf_like) {
        // y = (B/a) t - (rho h a (b.t)/Sf) k, pi = Gamma p rho h (b.t) k^2/Sf
        const R Sf = s.rh * a * a - s.gp * k2;
        const R cf = bt == (R)0 ? (R)0 : s.rh * bt * rcp<R>(Sf);
        const R r = Bx * rcp<R>(a);
        const R pk = cf * k2;
        q.p = s.gp * pk;
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            y[m] = r * tv[m] - cf * a * kv[m];
            z[m] = r * y[m] + s.b[m] * pk;
        }
    } else {
        // y = a (-k + B (rho h - Gamma p) k^2 (b.t)/(rho h Delta t^2) t), pi = Gamma p k^2
        const R De = s.e * a * a - Bx * Bx;
        const R cf = bt == (R)0 ? (R)0 : Bx * (s.rh - s.gp) * k2 * bt * rcp<R>(s.rh * De * mdot<R>(tv, tv));
        q.p = s.gp * k2;
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const R yy = cf * tv[m] - kv[m];
            y[m] = a * yy;
            z[m] = Bx * yy + s.b[m] * k2;
        }
    }
    const R by = mdot<R>(s.b, y);
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        q.u[m] = y[m];
        q.b[m] = z[m] + by * s.u[m];
    }
    mhd_scale<R>(s, q);
}

// The six waves' |a| and the frame data shared by their vectors.
template <typename R>
struct MhdSix {
    R t[6], sqe, c[2][4];
    bool alf[2];   // per side: the fast wave is the Alfven-like one
};

template <typename R>
__device__ __forceinline__ void mhd_six(const MhdBase<R> &s, MhdSix<R> &x, R lam[6])
{
    x.sqe = sq_rt<R>(s.e);
    for (int side = 0; side < 2; ++side) {
        const int sg = side == 0 ? 1 : -1;
        R tA, ts, tf;
        mhd_side<R>(s, x.sqe, sg, true, tA, ts, tf);
        const int o = side == 0 ? 0 : 5, d = side == 0 ? 1 : -1;
        x.t[o] = tf;
        x.t[o + d] = tA;
        x.t[o + 2 * d] = ts;
        const R a = (R)sg * tA, la = s.v1 - a * s.iW;
        x.alf[side] = s.rh * a * a > s.gp * (((R)1 - la) * ((R)1 + la) + a * a);
        // b along k (|b_t| at rounding level) or no field: the plane normal to
        // k spanned from a coordinate axis, the same for the side's waves
        R sv[4];
        mcross<R>(s.u, la, s.b, sv);
        const R bt2 = mdot<R>(sv, sv);
        const R A = s.u[0] - la * s.u[1];
        if (bt2 > (R)(sizeof(R) == 4 ? 1.0e-10 : 1.0e-22) * s.b2 * A * A) {
            for (int m = 0; m < 4; ++m) x.c[side][m] = s.b[m];
        } else {
            x.c[side][0] = x.c[side][1] = x.c[side][3] = (R)0;
            x.c[side][2] = (R)1;
        }
    }
#pragma unroll
    for (int m = 0; m < 6; ++m) lam[m] = m < 3 ? s.v1 - x.t[m] * s.iW : s.v1 + x.t[m] * s.iW;
}

template <typename R>
__device__ __forceinline__ void mhd_six_wave(const MhdBase<R> &s, const MhdSix<R> &x, int m, MhdWave<R> &q)
{
    const int side = m < 3 ? 0 : 1, kind = m < 3 ? m : 5 - m;   // 0 fast, 1 Alfven, 2 slow
    const bool alf_like = kind == 0 ? x.alf[side] : !x.alf[side];
    mhd_wave<R>(s, x.sqe, kind, side == 0 ? 1 : -1, x.t[m], alf_like, x.c[side], q);
}

}  // namespace esmm

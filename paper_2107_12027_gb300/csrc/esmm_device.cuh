// esmm_device.cuh -- device arithmetic of the ES adaptive moving-mesh scheme
// (Duan & Tang, arXiv 2107.12027), 2D RHD, templated on the working precision
// R (double for the FP64 form, float for the mixed form).  The primitive
// recovery is always FP64; the jumps of the logarithmic mean are formed in FP64, or in
// FP32 from values carried with their FP64 rest (LmV).
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <type_traits>

#include "esmm_conv.h"

namespace esmm {

constexpr int GH = 3;        // ghost layers of the padded node arrays
constexpr int PMAX = 3;      // largest supported p
// Node quantities stored per padded node (FP64, structure of arrays).
enum {
    Q_RHO = 0, Q_P, Q_BETA, Q_UX, Q_UY, Q_W, Q_LNR, Q_LNB,
    Q_M00, Q_M01, Q_M10, Q_M11, Q_MT0, Q_MT1, NQ
};
// FP32 copies of the node quantities that the mixed form's flux kernels read
// (written by the FP64 node pass, so that no flux kernel converts a double).
enum {
    Q32_R = 0, Q32_B, Q32_UX, Q32_UY, Q32_W, Q32_LNR, Q32_LNB,
    Q32_M00, Q32_M01, Q32_M10, Q32_M11, Q32_MT0, Q32_MT1, NQ32
};

struct Geom {
    int nx, ny;       // interior nodes
    int px, py;       // padded extents nx + 2 GH, ny + 2 GH
    long long P;      // px * py
    long long N;      // nx * ny
    int bc0, bc1;     // 0 periodic, 1 outflow
    double per0, per1;
    int own0, own1;   // rows j in [own0, own1) take part in the reductions
                      // (0, ny except on a slab of a decomposed grid)
};

// a node in the rows whose values the problem's reductions collect
__device__ __forceinline__ bool owned_row(const Geom &g, int j) { return j >= g.own0 && j < g.own1; }

// One problem of a batch: its geometry and the offsets of its slices in the
// concatenated arrays (on: node arrays, in units of nodes; op: padded-node
// arrays, in units of padded nodes).
struct ProbDesc {
    Geom g;
    long long on, op;
};

// Problem addressing of a launch: a single problem passed by value (tiles ==
// nullptr), or a device table of problems with a map from block to
// (problem, block within the problem), so that no block spans two problems.
struct ProbArg {
    const ProbDesc *pd;
    const int2 *tiles;
    ProbDesc one;
};

__device__ __forceinline__ int locate(const ProbArg &pa, ProbDesc &D, long long &local_block)
{
    if (pa.tiles) {
        int2 t = pa.tiles[blockIdx.x];
        D = pa.pd[t.x];
        local_block = t.y;
        return t.x;
    }
    D = pa.one;
    local_block = blockIdx.x;
    return 0;
}

// locate() for tile t of a strided launch (the block -> tile map of a
// batch, or tile t itself)
__device__ __forceinline__ int locate_tile(const ProbArg &pa, long long t, ProbDesc &D, long long &local_block)
{
    if (pa.tiles) {
        int2 tt = pa.tiles[t];
        D = pa.pd[tt.x];
        local_block = tt.y;
        return tt.x;
    }
    D = pa.one;
    local_block = t;
    return 0;
}

// The site (i, j) of thread threadIdx.x in tile lb of a sweep of direction
// dir over sites with ext extra positions before the first node along the
// sweep (p node pairs, 1 interface).  tx = 0: tiles are flat runs along the
// sweep's storage order; tx > 0: tiles of tx sites along x_1 by
// blockDim.x / tx along x_2.  false: no site (ragged tile).
__device__ __forceinline__ bool sweep_site(const Geom &g, int dir, int ext, int tx, long long lb, int &i, int &j)
{
    const int nd = dir == 0 ? g.nx : g.ny, no = dir == 0 ? g.ny : g.nx;
    if (tx == 0) {
        const long long idx = lb * blockDim.x + threadIdx.x;
        if (idx >= (long long)(nd + ext) * no) return false;
        if (dir == 0) { j = (int)(idx / (nd + ext)); i = (int)(idx % (nd + ext)) - ext; }
        else { i = (int)(idx % no); j = (int)(idx / no) - ext; }
        return true;
    }
    const int ty = blockDim.x / tx;
    const int Ei = dir == 0 ? nd + ext : no, Ej = dir == 0 ? no : nd + ext;
    const long long nbi = (Ei + tx - 1) / tx;
    const int ii = (int)(lb % nbi) * tx + (int)threadIdx.x % tx;
    const int jj = (int)(lb / nbi) * ty + (int)threadIdx.x / tx;
    if (ii >= Ei || jj >= Ej) return false;
    i = dir == 0 ? ii - ext : ii;
    j = dir == 0 ? jj : jj - ext;
    return true;
}

// FP64 <-> FP32 conversions on the integer pipes (esmm_conv.h), equal bit
// for bit to the hardware conversions, which issue on the FP64 pipe
template <typename T>
__device__ __forceinline__ T from_f64(double x);
template <>
__device__ __forceinline__ double from_f64<double>(double x) { return x; }
template <>
__device__ __forceinline__ float from_f64<float>(double x) { return d2f_int(x); }
__device__ __forceinline__ double to_f64(double x) { return x; }
__device__ __forceinline__ double to_f64(float x) { return f2d_int(x); }

struct Phys {
    double gamma;
    double gm1i;      // 1 / (Gamma - 1), once per launch
    double igg;       // (Gamma - 1) / Gamma
    double eps;       // WENO epsilon
    double ln_thr;    // log-mean series switch on ((b-a)/(b+a))^2
    double sign_tol;  // relative size below which [[V~]] counts as zero
    double alpha[PMAX];
    int p, w;
};

__host__ __device__ __forceinline__ long long pidx(const Geom &g, int i, int j)
{
    return (long long)(j + GH) * g.px + (i + GH);
}

__device__ __forceinline__ int wrapi(int a, int n) { int r = a % n; return r < 0 ? r + n : r; }
__device__ __forceinline__ int floordivi(int a, int n) { return a >= 0 ? a / n : -((-a + n - 1) / n); }
__device__ __forceinline__ int clampi(int a, int lo, int hi) { return a < lo ? lo : (a > hi ? hi : a); }

// Boundary data: periodic wrap or zero-gradient copy.
__device__ __forceinline__ long long data_src(const Geom &g, int i, int j)
{
    int ii = g.bc0 == 0 ? wrapi(i, g.nx) : clampi(i, 0, g.nx - 1);
    int jj = g.bc1 == 0 ? wrapi(j, g.ny) : clampi(j, 0, g.ny - 1);
    return (long long)jj * g.nx + ii;
}

// Boundary mesh: periodic wrap plus the period (shift = 1 for coordinates,
// 0 for velocities), or linear extrapolation of the two boundary nodes.
__device__ __forceinline__ double mesh_along_i(const Geom &g, const double *a, int i, int j, int comp, int shift)
{
    const double *row = a + (long long)comp * g.N + (long long)j * g.nx;
    if (g.bc0 == 0) {
        double s = (shift && comp == 0) ? floordivi(i, g.nx) * g.per0 : 0.0;
        return row[wrapi(i, g.nx)] + s;
    }
    if (i < 0) { double a0 = row[0], a1 = row[1]; return a0 + i * (a1 - a0); }
    if (i >= g.nx) { double a0 = row[g.nx - 1], a1 = row[g.nx - 2]; return a0 + (i - (g.nx - 1)) * (a0 - a1); }
    return row[i];
}

__device__ __forceinline__ double mesh_at(const Geom &g, const double *a, int i, int j, int comp, int shift)
{
    if (g.bc1 == 0) {
        double s = (shift && comp == 1) ? floordivi(j, g.ny) * g.per1 : 0.0;
        return mesh_along_i(g, a, i, wrapi(j, g.ny), comp, shift) + s;
    }
    if (j < 0) {
        double a0 = mesh_along_i(g, a, i, 0, comp, shift), a1 = mesh_along_i(g, a, i, 1, comp, shift);
        return a0 + j * (a1 - a0);
    }
    if (j >= g.ny) {
        double a0 = mesh_along_i(g, a, i, g.ny - 1, comp, shift), a1 = mesh_along_i(g, a, i, g.ny - 2, comp, shift);
        return a0 + (j - (g.ny - 1)) * (a0 - a1);
    }
    return mesh_along_i(g, a, i, j, comp, shift);
}

// ---------------------------------------------------------------------------
// Dual number a + b eps (eps^2 = 0): the flux arithmetic below is templated on
// its working type, and evaluating it on duals seeded at one input gives the
// derivative of every output with respect to that input.  The adjoint kernels
// use this for the interface state and for the second derivatives of (U, V, F).
struct dual {
    double v, d;
    __host__ __device__ dual() {}
    __host__ __device__ constexpr dual(double a) : v(a), d(0.0) {}
    __host__ __device__ constexpr dual(double a, double b) : v(a), d(b) {}
};
__device__ __forceinline__ dual operator+(dual a, dual b) { return dual(a.v + b.v, a.d + b.d); }
__device__ __forceinline__ dual operator-(dual a, dual b) { return dual(a.v - b.v, a.d - b.d); }
__device__ __forceinline__ dual operator-(dual a) { return dual(-a.v, -a.d); }
__device__ __forceinline__ dual operator*(dual a, dual b) { return dual(a.v * b.v, a.d * b.v + a.v * b.d); }
__device__ __forceinline__ dual operator/(dual a, dual b)
{
    double r = __drcp_rn(b.v);
    double q = a.v * r;
    return dual(q, (a.d - q * b.d) * r);
}
__device__ __forceinline__ dual operator+(dual a, double b) { return dual(a.v + b, a.d); }
__device__ __forceinline__ dual operator+(double a, dual b) { return dual(a + b.v, b.d); }
__device__ __forceinline__ dual operator-(dual a, double b) { return dual(a.v - b, a.d); }
__device__ __forceinline__ dual operator-(double a, dual b) { return dual(a - b.v, -b.d); }
__device__ __forceinline__ dual operator*(dual a, double b) { return dual(a.v * b, a.d * b); }
__device__ __forceinline__ dual operator*(double a, dual b) { return dual(a * b.v, a * b.d); }
__device__ __forceinline__ dual operator/(dual a, double b)
{
    const double r = __drcp_rn(b);
    return dual(a.v * r, a.d * r);
}
__device__ __forceinline__ dual operator/(double a, dual b) { return dual(a) / b; }
__device__ __forceinline__ dual &operator+=(dual &a, dual b) { a = a + b; return a; }
__device__ __forceinline__ dual &operator-=(dual &a, dual b) { a = a - b; return a; }
__device__ __forceinline__ dual &operator*=(dual &a, dual b) { a = a * b; return a; }
__device__ __forceinline__ double val(double x) { return x; }
__device__ __forceinline__ float val(float x) { return x; }
__device__ __forceinline__ double val(dual x) { return x.v; }

// The FP32 dual number (directional derivatives inside the FP32 bulk form).
// FP64 constants are rounded to FP32 before they meet an fdual, so no FP64
// arithmetic runs on its values.
struct fdual {
    float v, d;
    __host__ __device__ fdual() {}
    __host__ __device__ constexpr fdual(float a) : v(a), d(0.0f) {}
    __host__ __device__ constexpr fdual(float a, float b) : v(a), d(b) {}
};
__device__ __forceinline__ fdual operator+(fdual a, fdual b) { return fdual(a.v + b.v, a.d + b.d); }
__device__ __forceinline__ fdual operator-(fdual a, fdual b) { return fdual(a.v - b.v, a.d - b.d); }
__device__ __forceinline__ fdual operator-(fdual a) { return fdual(-a.v, -a.d); }
__device__ __forceinline__ fdual operator*(fdual a, fdual b) { return fdual(a.v * b.v, a.d * b.v + a.v * b.d); }
__device__ __forceinline__ fdual operator/(fdual a, fdual b)
{
    float r = __frcp_rn(b.v);
    float q = a.v * r;
    return fdual(q, (a.d - q * b.d) * r);
}
__device__ __forceinline__ fdual operator+(fdual a, double b) { return fdual(a.v + (float)b, a.d); }
__device__ __forceinline__ fdual operator+(double a, fdual b) { return fdual((float)a + b.v, b.d); }
__device__ __forceinline__ fdual operator-(fdual a, double b) { return fdual(a.v - (float)b, a.d); }
__device__ __forceinline__ fdual operator-(double a, fdual b) { return fdual((float)a - b.v, -b.d); }
__device__ __forceinline__ fdual operator*(fdual a, double b) { return fdual(a.v * (float)b, a.d * (float)b); }
__device__ __forceinline__ fdual operator*(double a, fdual b) { return fdual((float)a * b.v, (float)a * b.d); }
__device__ __forceinline__ fdual operator/(fdual a, double b) { return a / fdual((float)b); }
__device__ __forceinline__ fdual operator/(double a, fdual b) { return fdual((float)a) / b; }
__device__ __forceinline__ fdual &operator+=(fdual &a, fdual b) { a = a + b; return a; }
__device__ __forceinline__ fdual &operator-=(fdual &a, fdual b) { a = a - b; return a; }

// Hyper-dual number v + a e1 + b e2 + ab e1 e2 (e1^2 = e2^2 = 0): e1 carries a
// Jacobian image direction, e2 the adjoint's seeded state direction, and ab
// the mixed second derivative.  Used for the images of the RMHD
// eigen-system inside the adjoint.
struct hdual {
    double v, a, b, ab;
    __host__ __device__ hdual() {}
    __host__ __device__ constexpr hdual(double x) : v(x), a(0.0), b(0.0), ab(0.0) {}
    __host__ __device__ constexpr hdual(double x, double a_, double b_, double ab_) : v(x), a(a_), b(b_), ab(ab_) {}
};
__device__ __forceinline__ hdual operator+(hdual x, hdual y) { return hdual(x.v + y.v, x.a + y.a, x.b + y.b, x.ab + y.ab); }
__device__ __forceinline__ hdual operator-(hdual x, hdual y) { return hdual(x.v - y.v, x.a - y.a, x.b - y.b, x.ab - y.ab); }
__device__ __forceinline__ hdual operator-(hdual x) { return hdual(-x.v, -x.a, -x.b, -x.ab); }
__device__ __forceinline__ hdual operator*(hdual x, hdual y)
{
    return hdual(x.v * y.v, x.a * y.v + x.v * y.a, x.b * y.v + x.v * y.b,
                 x.ab * y.v + x.a * y.b + x.b * y.a + x.v * y.ab);
}
// f(x) for a scalar function with value f, first and second derivatives f1, f2 at x.v
__device__ __forceinline__ hdual hchain(hdual x, double f, double f1, double f2)
{
    return hdual(f, f1 * x.a, f1 * x.b, f1 * x.ab + f2 * x.a * x.b);
}
__device__ __forceinline__ hdual hrcp(hdual x)
{
    double r = __drcp_rn(x.v);
    return hchain(x, r, -r * r, 2.0 * r * r * r);
}
__device__ __forceinline__ hdual operator/(hdual x, hdual y) { return x * hrcp(y); }
__device__ __forceinline__ hdual operator+(hdual x, double y) { return hdual(x.v + y, x.a, x.b, x.ab); }
__device__ __forceinline__ hdual operator+(double x, hdual y) { return hdual(x + y.v, y.a, y.b, y.ab); }
__device__ __forceinline__ hdual operator-(hdual x, double y) { return hdual(x.v - y, x.a, x.b, x.ab); }
__device__ __forceinline__ hdual operator-(double x, hdual y) { return hdual(x - y.v, -y.a, -y.b, -y.ab); }
__device__ __forceinline__ hdual operator*(hdual x, double y) { return hdual(x.v * y, x.a * y, x.b * y, x.ab * y); }
__device__ __forceinline__ hdual operator*(double x, hdual y) { return hdual(x * y.v, x * y.a, x * y.b, x * y.ab); }
__device__ __forceinline__ hdual operator/(hdual x, double y) { return x * __drcp_rn(y); }
__device__ __forceinline__ hdual operator/(double x, hdual y) { return x * hrcp(y); }

// the dual number over a working precision (hdual over dual)
template <typename R> struct DualOf { using type = dual; };
template <> struct DualOf<float> { using type = fdual; };
template <> struct DualOf<dual> { using type = hdual; };
// an image seed: value w moved along direction d (for hdual: w, d are duals
// whose .d parts are the seeded state direction and d's derivative along it)
__device__ __forceinline__ dual img_seed(double w, double d) { return dual(w, d); }
__device__ __forceinline__ fdual img_seed(float w, float d) { return fdual(w, d); }
__device__ __forceinline__ hdual img_seed(dual w, dual d) { return hdual(w.v, d.v, w.d, d.d); }
// the image part of a seeded result, in the working precision
__device__ __forceinline__ double img_part(dual x) { return x.d; }
__device__ __forceinline__ float img_part(fdual x) { return x.d; }
__device__ __forceinline__ dual img_part(hdual x) { return dual(x.a, x.ab); }

// type of the log-mean arguments: FP64 for the FP64 and FP32-bulk forms
template <typename R> struct LogT { using type = double; };
template <> struct LogT<dual> { using type = dual; };

template <typename R> __device__ __forceinline__ R rsq(R x);
template <> __device__ __forceinline__ double rsq<double>(double x) { return rsqrt(x); }
template <> __device__ __forceinline__ float rsq<float>(float x) { return rsqrtf(x); }
template <> __device__ __forceinline__ dual rsq<dual>(dual x)
{
    double r = rsqrt(x.v);
    return dual(r, -0.5 * r * r * r * x.d);
}
template <typename R> __device__ __forceinline__ R sq_rt(R x);
template <> __device__ __forceinline__ double sq_rt<double>(double x) { return sqrt(x); }
template <> __device__ __forceinline__ float sq_rt<float>(float x) { return sqrtf(x); }
template <> __device__ __forceinline__ dual sq_rt<dual>(dual x)
{
    double r = sqrt(x.v);
    return dual(r, 0.5 * x.d / r);
}
template <> __device__ __forceinline__ fdual sq_rt<fdual>(fdual x)
{
    float r = sqrtf(x.v);
    return fdual(r, 0.5f * x.d * __frcp_rn(r));
}
template <> __device__ __forceinline__ hdual sq_rt<hdual>(hdual x)
{
    double r = sqrt(x.v);
    double r1 = 0.5 / r;
    return hchain(x, r, r1, -0.5 * r1 / x.v);
}
// reciprocal (IEEE round-to-nearest) and a square root of a positive value
// through the reciprocal square root: on GB300 both are cheaper than the
// FP64 quotient and square root
template <typename R> __device__ __forceinline__ R rcp(R x);
template <> __device__ __forceinline__ double rcp<double>(double x) { return __drcp_rn(x); }
template <> __device__ __forceinline__ float rcp<float>(float x) { return __frcp_rn(x); }
template <> __device__ __forceinline__ dual rcp<dual>(dual x)
{
    double r = __drcp_rn(x.v);
    return dual(r, -r * r * x.d);
}
template <> __device__ __forceinline__ fdual rcp<fdual>(fdual x)
{
    float r = __frcp_rn(x.v);
    return fdual(r, -r * r * x.d);
}
template <> __device__ __forceinline__ hdual rcp<hdual>(hdual x) { return hrcp(x); }
template <> __device__ __forceinline__ fdual rsq<fdual>(fdual x)
{
    float r = rsqrtf(x.v);
    return fdual(r, -0.5f * r * r * r * x.d);
}
template <> __device__ __forceinline__ hdual rsq<hdual>(hdual x)
{
    // x^-1/2 and its first two derivatives
    double r = rsqrt(x.v), ir = __drcp_rn(x.v);
    return hchain(x, r, -0.5 * r * ir, 0.75 * r * ir * ir);
}
template <typename R> __device__ __forceinline__ R sqrt_pos(R x) { return x * rsq<R>(x); }

// a b + c in one rounding, and a - b not contracted with what forms or uses them (left to
// itself the compiler contracts by what it sees in a basic block, so that two kernels
// inlining one function may round differently)
template <typename R> __device__ __forceinline__ R fma_(R a, R b, R c) { return a * b + c; }
template <> __device__ __forceinline__ double fma_<double>(double a, double b, double c) { return __fma_rn(a, b, c); }
template <> __device__ __forceinline__ float fma_<float>(float a, float b, float c) { return __fmaf_rn(a, b, c); }

template <typename R> __device__ __forceinline__ R sub_(R a, R b) { return a - b; }
template <> __device__ __forceinline__ double sub_<double>(double a, double b) { return __dsub_rn(a, b); }
template <> __device__ __forceinline__ float sub_<float>(float a, float b) { return __fsub_rn(a, b); }

// Reciprocal of a non-zero and reciprocal square root of a positive normal finite
// number, within about an ulp: the hardware's first approximation (error below 2^-20
// in FP64, 2^-22 in FP32) and one correction by the series of 1/(1-e) and
// (1-e)^-1/2 in its residual e (Householder's iteration of third order in FP64, of
// second order in FP32).  In FP64 that is 3 and 5 FP64 instructions, against about 7
// and 10 of the correctly rounded reciprocal and of rsqrt, whose special cases (zero,
// infinite, subnormal arguments) these leave out: here they give a NaN.
// (Compiled for the host, the approximations are IEEE quotients on the hardware's domain:
// subnormal arguments and results count as zero.)
#if defined(__CUDA_ARCH__)
__device__ __forceinline__ double approx_rcp(double x)
{
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    return r;
}
__device__ __forceinline__ float approx_rcp(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ double approx_rsq(double x)
{
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    return y;
}
#else
template <typename R> inline R ftz_(R x)
{
    const R tiny = sizeof(R) == 4 ? (R)1.17549435e-38f : (R)2.2250738585072014e-308;
    return x < tiny && x > -tiny ? x * (R)0 : x;
}
template <typename R> inline R approx_rcp(R x) { return ftz_<R>((R)1 / ftz_<R>(x)); }
inline double approx_rsq(double x) { return 1.0 / sqrt(ftz_<double>(x)); }
#endif
template <typename R> __device__ __forceinline__ R qrcp(R x) { return rcp<R>(x); }
template <typename R> __device__ __forceinline__ R qrsq(R x) { return rsq<R>(x); }
template <> __device__ __forceinline__ double qrcp<double>(double x)
{
    const double r = approx_rcp(x), e = __fma_rn(-x, r, 1.0);
    return __fma_rn(r, __fma_rn(e, e, e), r);
}
template <> __device__ __forceinline__ float qrcp<float>(float x)
{
    const float r = approx_rcp(x);
    return __fmaf_rn(r, __fmaf_rn(-x, r, 1.0f), r);
}
template <> __device__ __forceinline__ double qrsq<double>(double x)
{
    const double y = approx_rsq(x), e = __fma_rn(-__dmul_rn(x, y), y, 1.0);
    return __fma_rn(__dmul_rn(y, e), __fma_rn(0.375, e, 0.5), y);
}
// sqrt(x) as x qrsq(x) where that holds, sqrt's own value for 0, subnormal, infinite and
// negative x
__device__ __forceinline__ double qsqrt(double x)
{
    return (conv_bits64(x) >> 52) - 1ull < 0x7feull ? x * qrsq<double>(x) : sqrt(x);
}
// acoustic speeds along a normal with velocity vn; iden = 1/(1 - v^2 c^2) (their root is 0 where
// rounding leaves v^2 = 1)
__device__ __forceinline__ void rhd_speeds(double v2, double c2, double cs, double iden, double vn, double &lm, double &lp)
{
    const double disc = qsqrt((1.0 - v2) * (1.0 - v2 * c2 - vn * vn * (1.0 - c2)));
    lm = (vn * (1.0 - c2) - cs * disc) * iden;
    lp = (vn * (1.0 - c2) + cs * disc) * iden;
}
template <typename R> __device__ __forceinline__ R fab(R x);
template <> __device__ __forceinline__ double fab<double>(double x) { return fabs(x); }
template <> __device__ __forceinline__ float fab<float>(float x) { return fabsf(x); }
template <> __device__ __forceinline__ dual fab<dual>(dual x) { return x.v < 0.0 ? -x : x; }
// larger of two values (the derivative follows the selected argument)
__device__ __forceinline__ double vmax(double a, double b) { return fmax(a, b); }
__device__ __forceinline__ float vmax(float a, float b) { return fmaxf(a, b); }
__device__ __forceinline__ dual vmax(dual a, dual b) { return a.v >= b.v ? a : b; }

// Logarithmic mean [[a]]/[[ln a]] and its reciprocal from FP64 node values
// and their FP64 logarithms.  Near-equal arguments, ((b-a)/(b+a))^2 < thr, use
// the Ismail-Roe series in FP64: mean = (a+b)/(2 F), F = 1 + u/3 + u^2/5 + u^3/7.
template <typename R, typename T>
__device__ __forceinline__ void logmean(T a, T b, T la, T lb, double thr, R &mean, R &inv_mean)
{
    T d = b - a, s = b + a;
    if (val(d * d) < val(thr * s * s)) {
        // (two reciprocals for the three quotients: each product is within
        // an ulp of the quotient it stands for)
        T is = rcp<T>(s);
        T r = d * is, u = r * r;
        T F = 1.0 + u * (1.0 / 3.0 + u * (1.0 / 5.0 + u * (1.0 / 7.0)));
        mean = (R)(0.5 * s * rcp<T>(F));
        inv_mean = (R)(2.0 * F * is);
    } else {
        R dn = (R)d, dl = (R)(lb - la);
        mean = dn * rcp<R>(dl);
        inv_mean = dl * rcp<R>(dn);
    }
}

// ---------------------------------------------------------------------------
// Conservative -> primitive recovery (FP64 in every form).  The root in p of
//   f(p) = (G-1)/G ((E+p)(1-v^2) - D sqrt(1-v^2)) - p,  v = |m|/(E+p).
// An FP32 Newton iteration (c2p_estimate, off the FP64 pipe) gives p to about 1e-7 (E + p);
// one FP64 step of third order (Halley's; the curvature in FP32) then lands on the root
// to rounding, in any units (the FP32 parts work over the power of two below E): it is the last where it is below 3e-6 of E + p - |m|, the length on
// which f bends, and its second-order part below 3e-6 of it, which leaves the next
// term under 1e-11 of the step.  Where that fails three times (an estimate that failed,
// states at the edge of the admissible set) c2p_loop starts over: FP64 Newton safeguarded by bisection on [0, (G-1)E],
// stopping when a step moves p by at most 1e-15 (E + p), the resolution of E + p from
// which f is evaluated, or when |f| <= 2e-15 (E + p), f's own rounding level (where df/dp
// is small, steps at that level exceed the first bound and the loop would bisect).
// p0 is a warm start (ignored when outside the bracket).  W receives the Lorentz factor
// 1/sqrt(1-v^2) (1 for a non-admissible state).  Returns 0, 1 for a non-admissible state,
// 2 when the iteration cap is hit.  gg = (Gamma - 1)/Gamma, which a launch can pass in
// (one division per launch, not per node).
// Bound: the FP64 pipe (the padded nodes of a large grid) and the chain of dependent
// FP64 operations (a small one); ~70 FP64 instructions against ~45 per step of the loop
// alone, two to four steps from a warm start and eight to ten from a cold one.  Measured
// (64 registers a thread): mixed 400^2 steps 1.22 -> 1.15 ms, the mixed batch 88.9 -> 81.6 ms,
// one 64^2 right-hand side from a cold start 37.5 -> 35.3 us, 64^2 steps 1.65 -> 1.66 ms.
// Against extended precision p is 2 times closer in the median and 10 in the worst percent
// (the loop stops within 2e-15 (E + p) of a root).
__device__ __forceinline__ float c2p_estimate(float gg, float D, float S2, float S, float EmS, float E, float hi0, float p0)
{
    float lo = 0.0f, hi = hi0, p = p0;
#pragma unroll 1
    for (int it = 0; it < 24; ++it) {
        const float Ep = E + p, r = __frcp_rn(Ep), iW2 = (EmS + p) * (Ep + S) * (r * r), rs = rsqrtf(iW2), v2 = S2 * r * r;
        const float f = gg * (Ep * iW2 - D * (iW2 * rs)) - p, df = gg * (1.0f + v2 - D * v2 * r * rs) - 1.0f;
        if (f > 0.0f) lo = p; else hi = p;
        float pn = p - f * __frcp_rn(df);
        // (a step this small ends the iteration: the next would be its square; the bracket,
        // whose ends FP32 rounding moves, has no say in it)
        const bool done = fabsf(pn - p) <= 2.0e-4f * (EmS + p);
        if (!done && !(pn > lo && pn < hi)) pn = 0.5f * (lo + hi);
        p = pn;
        if (done) break;
    }
    return p;
}

static __device__ __noinline__ int c2p_loop(double gg, double D, double S2, double S, double E, double hi, double &pc)
{
    double lo = 0.0;
#pragma unroll 1
    for (int it = 0; it < 200; ++it) {
        const double Ep = E + pc, r = __drcp_rn(Ep);
        const double iW2 = (Ep - S) * (Ep + S) * r * r;    // 1 - v^2
        const double rs = rsqrt(iW2);
        const double v2 = S2 * r * r;
        const double f = gg * (Ep * iW2 - D * (iW2 * rs)) - pc;
        if (fabs(f) <= 2.0e-15 * (E + pc)) return 0;   // residual at rounding level
        if (f > 0.0) lo = pc; else hi = pc;
        const double df = gg * (1.0 + v2 - D * v2 * r * rs) - 1.0;
        double pn = pc - f * f2d_int(__frcp_rn(d2f_int(df)));   // (the slope only steers the step)
        if (!(pn > lo && pn < hi)) pn = 0.5 * (lo + hi);
        const bool done = fabs(pn - pc) <= 1.0e-15 * (E + pn);
        pc = pn;
        if (done) return 0;
    }
    return 2;
}

__device__ __forceinline__ int cons2prim_gg(double gam, double gg, double D, double mx, double my, double E,
                                            double p0, double &rho, double &vx, double &vy, double &p, double &W)
{
    const double S2 = mx * mx + my * my;
    rho = 0.0; vx = 0.0; vy = 0.0; p = 0.0; W = 1.0;
    if (!(D > 0.0) || !(E * E > D * D + S2) || !(E > 0.0)) return 1;
    double S;
    if (conv_bits64(S2) >> 52 > 64u) {   // (no subnormal reciprocal root)
        const double y = qrsq<double>(S2), S_ = S2 * y;
        S = __fma_rn(__fma_rn(-S_, S_, S2), 0.5 * y, S_);
    } else {
        S = sqrt(S2);
    }
    const double hi = (gam - 1.0) * E, EmS = E - S;
    const double pw = (p0 > 0.0 && p0 < hi) ? p0 : 0.5 * hi;
    const int k = binade(E);   // the FP32 parts take every quantity over 2^k
    const float ggf = d2f_int(gg), Df = d2f_scaled(D, k), EmSf = d2f_scaled(EmS, k), Sf = d2f_scaled(S, k);
    const float pf = c2p_estimate(ggf, Df, Sf * Sf, Sf, EmSf, d2f_scaled(E, k), d2f_scaled(hi, k), d2f_scaled(pw, k));
    double pc = f2d_scaled(pf, k);
    int st = 0;
    bool ok = false;
#pragma unroll 1
    for (int it = 0; it < 3; ++it) {   // (a second step where the estimate was poor)
        const double Ep = E + pc, r = qrcp<double>(Ep), iW2 = (EmS + pc) * (Ep + S) * (r * r), rs = qrsq<double>(iW2);
        const double v2 = S2 * (r * r), Dw = D * rs;
        const double f = gg * (Ep * iW2 - Dw * iW2) - pc, df = gg * (1.0 + v2 - Dw * (v2 * r)) - 1.0;
        const double dp = f * qrcp<double>(df);
        const float rf = d2f_scaled(r, -k), vf = d2f_int(v2), sf = d2f_int(rs), dpf = d2f_scaled(dp, k);
        const float a = vf * rf, f2 = ggf * (Df * sf * (3.0f * a * rf + a * a * (sf * sf)) - 2.0f * a);
        const float eta = 0.5f * f2 * dpf * __frcp_rn(d2f_int(df));
        ok = fabsf(dpf) <= 3.0e-6f * (EmSf + d2f_scaled(pc, k)) && fabsf(eta) <= 3.0e-6f;
        const double pn = pc - __fma_rn(dp, f2d_int(eta), dp);
        if (!(d2f_scaled(pn, k) > 0.0f) || !(fabsf(eta) <= 0.1f)) {
            ok = false;
            break;
        }
        pc = pn;
        if (ok) break;
    }
    if (!ok) {
        pc = pw;
        st = c2p_loop(gg, D, S2, S, E, hi, pc);
    }
    const double Ep = E + pc, r = ok ? qrcp<double>(Ep) : __drcp_rn(Ep), iW2 = (EmS + pc) * (Ep + S) * (r * r);
    W = ok ? qrsq<double>(iW2) : rsqrt(iW2);
    rho = D * (iW2 * W);
    vx = mx * r;
    vy = my * r;
    p = pc;
    return st;
}

__device__ __forceinline__ int cons2prim(double gam, double D, double mx, double my, double E,
                                         double p0, double &rho, double &vx, double &vy, double &p, double &W)
{
    return cons2prim_gg(gam, (gam - 1.0) / gam, D, mx, my, E, p0, rho, vx, vy, p, W);
}

// An argument of the log means: the value and its logarithm, in FP32 with the
// rest of the FP64 value, so that the jump of two near-equal values keeps FP32
// relative precision without FP64 arithmetic: (b.v - a.v) is exact within a factor 2
// of each other, and v + lo carries 48 bits.
template <typename R> struct LmV { R v, l; };
template <> struct LmV<float> { float v, lo, l; };
__device__ __forceinline__ LmV<float> lmv_f32(double x, float v, float l)
{
    LmV<float> a;
    a.v = v;
    a.lo = d2f_int(x - f2d_int(v));
    a.l = l;
    return a;
}
__device__ __forceinline__ float to_f32(double x) { return d2f_int(x); }
__device__ __forceinline__ float to_f32(float x) { return x; }

// Logarithmic mean (b - a)/(ln b - ln a) and its reciprocal; near-equal arguments,
// |b - a| < sqrt(thr) (a + b), by the Ismail-Roe series F = 1 + u/3 + u^2/5 + u^3/7 in
// u = ((b-a)/(b+a))^2: inverse 2F/(a+b), mean (a+b)/2 times the series of 1/F (their
// dropped terms are below u^4/9).  The switch is taken in FP32 where it holds the values
// (both branches hold at the switch; FP64 compares cost FP64-pipe slots).
template <typename R>
__device__ __forceinline__ void logmean2(const LmV<R> &a, const LmV<R> &b, double thr, R &mean, R &inv_mean)
{
    R d, s;
    bool near;
    if constexpr (std::is_same<R, float>::value) {
        d = (b.v - a.v) + (b.lo - a.lo);
        s = b.v + a.v;
        near = d * d < (float)thr * (s * s);
    } else {
        d = b.v - a.v;
        s = b.v + a.v;
        if constexpr (std::is_same<R, double>::value) {
            const float d32 = d2f_int(d), s32 = d2f_int(s);
            near = s32 > 1.0e-30f && s32 < 1.0e30f ? fabsf(d32) < sqrtf((float)thr) * s32 : d * d < thr * s * s;
        } else {
            near = val(d * d) < val(thr * s * s);
        }
    }
    if (near) {
        const R is = qrcp<R>(s), r = d * is, u = r * r;
        mean = (R)0.5 * s * ((R)1 + u * ((R)(-1.0 / 3.0) + u * ((R)(-4.0 / 45.0) + u * (R)(-44.0 / 945.0))));
        inv_mean = (R)2 * is * ((R)1 + u * ((R)(1.0 / 3.0) + u * ((R)(1.0 / 5.0) + u * (R)(1.0 / 7.0))));
    } else {
        const R dl = b.l - a.l;
        mean = d * qrcp<R>(dl);
        inv_mean = dl * qrcp<R>(d);
    }
}

// Node values of one two-point flux argument (the parameter variables).
template <typename R>
struct NodeV {
    LmV<R> rho, beta;
    R ux, uy, W;
};

// Curvilinear two-point EC flux of Sec. 3.1 for one node pair in direction k:
//   F~_k = 1/2 (mt_l + mt_r) U~ + sum_j 1/2 (M_kj,l + M_kj,r) F~_j,
// mt, mx, my the averaged metrics.  U~ is the paper's U~^RMHD at B = 0 and
// F~_j the matching RHD spatial flux:
//   U~_D = r_ln W,  U~_E = (alpha0 U~_D W + pm |u|^2)/Lam,
//   U~_m = (U~_E + pm) u/W,  F~_D,j = r_ln u_j,
//   F~_E,j = W (alpha0 r_ln + pm) u_j / Lam,  F~_m,j = F~_E,j u/W + pm e_j,
// with the arithmetic means r, b, u, W, pm = r/b, Lam = W^2 - |u|^2 and
// alpha0 = 1 + 1/((Gamma-1) b_ln).  Contracting with the metrics gives
//   out_D = r_ln (mt W + un), out_E = mt U~_E + Es,
//   out_m = u/W (mt (U~_E + pm) + Es) + pm (mx, my),
// un = mx u_x + my u_y, Es = W (alpha0 r_ln + pm) un / Lam.
template <typename R>
__device__ __forceinline__ void ec_pair(const NodeV<R> &l, const NodeV<R> &r, R mt, R mx, R my,
                                        R gm1inv, double thr, R out[4])
{
    R rln, irln, bln, ibln;
    logmean2<R>(l.rho, r.rho, thr, rln, irln);
    logmean2<R>(l.beta, r.beta, thr, bln, ibln);
    R half = (R)0.5;
    R Wm = half * (l.W + r.W);
    R uxm = half * (l.ux + r.ux);
    R uym = half * (l.uy + r.uy);
    R usq = uxm * uxm + uym * uym;
    R Lam = Wm * Wm - usq;
    R alpha0 = (R)1 + gm1inv * ibln;
    R pm = (l.rho.v + r.rho.v) * qrcp<R>(l.beta.v + r.beta.v);
    R rinv = qrcp<R>(Lam * Wm);
    R iLam = rinv * Wm;
    R iW = rinv * Lam;
    R UD = rln * Wm;
    R UE = (alpha0 * UD * Wm + pm * usq) * iLam;
    R un = mx * uxm + my * uym;
    R Es = Wm * (alpha0 * rln + pm) * un * iLam;
    R cm = (mt * (UE + pm) + Es) * iW;
    out[0] = rln * (mt * Wm + un);
    out[1] = uxm * cm + pm * mx;
    out[2] = uym * cm + pm * my;
    out[3] = mt * UE + Es;
}

// The jump (right minus left Jiang-Shu edge value) at one interface from the first
// differences D_k = V_{k+1} - V_k of its stencil.  WENO5, V0..V5 with the interface
// between V2 and V3: with the second differences t, the third differences d and the
// candidates of the left value q_0, q_a, q_b (q_a, q_b also the right value's),
//   q_0 - q_a = d_0/3,  q_b - q_a = d_1/6,  q_0' - q_b = -d_2/3,
// the weights a_k = d_k/(eps + b_k)^2 (multiplied through by the squared denominators)
// give left = q_a + (2 a_0 d_0 + a_2 d_1)/(6 sum a), and likewise on the right, so that
//   jump = (d_1 - (2 a_0' d_2 + a_2' d_1)/sum a' - (2 a_0 d_0 + a_2 d_1)/sum a)/6
// without the edge values themselves: ~60 operations against ~95, and no cancellation
// of the field's mean value (with the eigenvectors in closed form below, the FP32
// tolerance and the short reciprocals: the 400^2 FP64 step 5.50 -> 4.26 ms, the mixed one
// 1.25 -> 1.22 ms, one 64^2 right-hand side 44 -> 37 us).  Everything is scaled by 4 (eps4 = 4 eps, b_k of doubled
// first-derivative terms).  Sums of two products are written as the fused operation, so
// that every kernel that inlines this rounds them alike.
// FP32: the products of four e (up to 33 D^2 each, down to 4 eps) and a difference would leave the
// range from D ~ 2,600 up, and for eps below ~1e-10.  The weights are 1/e^2 there instead, by the
// hardware's reciprocals (within an ulp): as many instructions, and D to 1e8, eps down to 1e-19
// (400^2 mixed step 1.120 -> 1.108 ms).
template <typename R>
__device__ __forceinline__ void weno5_side(R e0, R e1, R e2, R d0, R d1, R &n, R &q)
{
    if constexpr (std::is_same<R, float>::value) {
        e0 = approx_rcp(e0); e1 = approx_rcp(e1); e2 = approx_rcp(e2);
        e0 *= e0; e1 *= e1; e2 *= e2;
        n = fma_<R>(2.0f, e0 * d0, 3.0f * (e2 * d1));
        q = qrcp<R>(fma_<R>(6.0f, e1, fma_<R>(3.0f, e2, e0)));
    } else {
        const R two = (R)2, three = (R)3, six = (R)6;
        e0 *= e0; e1 *= e1; e2 *= e2;
        n = e1 * fma_<R>(three, e0 * d1, two * (e2 * d0));
        q = qrcp<R>(fma_<R>(e2, fma_<R>(six, e0, e1), three * (e0 * e1)));
    }
}
template <typename R>
__device__ __forceinline__ R weno5_jump(R D0, R D1, R D2, R D3, R D4, R eps4)
{
    const R c = (R)(13.0 / 3.0), two = (R)2;
    const R t0 = D1 - D0, ta = D2 - D1, tb = D3 - D2, t5 = D4 - D3;
    const R d0 = t0 - ta, d1 = ta - tb, d2 = tb - t5;
    const R S0 = fma_<R>(c * t0, t0, eps4), Sa = fma_<R>(c * ta, ta, eps4), Sb = fma_<R>(c * tb, tb, eps4),
            S5 = fma_<R>(c * t5, t5, eps4);
    R nl, ql, nr, qr;
    {
        const R r0 = t0 + two * D1, r1 = D1 + D2, r2 = tb - two * D2;
        R e0 = fma_<R>(r0, r0, S0), e1 = fma_<R>(r1, r1, Sa), e2 = fma_<R>(r2, r2, Sb);
        weno5_side<R>(e0, e1, e2, d0, d1, nl, ql);
    }
    {
        const R r0 = t5 - two * D3, r1 = D2 + D3, r2 = ta + two * D2;
        R e0 = fma_<R>(r0, r0, S5), e1 = fma_<R>(r1, r1, Sb), e2 = fma_<R>(r2, r2, Sa);
        weno5_side<R>(e0, e1, e2, d2, d1, nr, qr);
    }
    return (d1 - fma_<R>(nl, ql, nr * qr)) * (R)(1.0 / 6.0);
}

// WENO3, V0..V3 with the interface between V1 and V2: left = q - w t_0/2, right =
// q - w' t_1/2 with q the mean of V1 and V2.
template <typename R>
__device__ __forceinline__ R weno3_jump(R D0, R D1, R D2, R eps)
{
    R e0 = fma_<R>(D0, D0, eps), e1 = fma_<R>(D1, D1, eps), e2 = fma_<R>(D2, D2, eps);
    e0 *= e0; e1 *= e1; e2 *= e2;
    const R w0 = e1 * qrcp<R>(fma_<R>((R)2, e0, e1)), w1 = e1 * qrcp<R>(fma_<R>((R)2, e2, e1));
    return (R)0.5 * fma_<R>(w0, D1 - D0, w1 * (D1 - D2));
}

// The two Jiang-Shu WENO5 edge values of one interface from its six stencil
// values V0..V5 (V2, V3 the interface's nodes): vm from V0..V4 (upwind
// left) and vp from V5..V1 (upwind right).  Each is
//   sum_k (d_k/(eps+b_k)^2) q_k / sum_k d_k/(eps+b_k)^2, d = (0.1, 0.6, 0.3),
// written with a single division by multiplying through by the three
// squared denominators.  The candidate values and second differences of the
// two middle candidate stencils, {V1, V2, V3} and {V2, V3, V4}, serve both
// reconstructions (left's 2nd and 3rd candidates are right's 3rd and 2nd)
// and are formed once.
template <typename R>
__device__ __forceinline__ void weno5_lr(R V0, R V1, R V2, R V3, R V4, R V5, R eps, R &vm, R &vp)
{
    const R c13_12 = (R)(13.0 / 12.0), c1_4 = (R)0.25, c1_6 = (R)(1.0 / 6.0);
    const R qa = (-V1 + (R)5 * V2 + (R)2 * V3) * c1_6;
    const R qb = ((R)2 * V2 + (R)5 * V3 - V4) * c1_6;
    const R ta = V1 - (R)2 * V2 + V3, tb = V2 - (R)2 * V3 + V4;
    const R sa = c13_12 * ta * ta, sb = c13_12 * tb * tb;
    {
        R q0 = ((R)2 * V0 - (R)7 * V1 + (R)11 * V2) * c1_6;
        R t0 = V0 - (R)2 * V1 + V2, r0 = V0 - (R)4 * V1 + (R)3 * V2;
        R r1 = V1 - V3, r2 = (R)3 * V2 - (R)4 * V3 + V4;
        R e0 = eps + c13_12 * t0 * t0 + c1_4 * r0 * r0;
        R e1 = eps + sa + c1_4 * r1 * r1;
        R e2 = eps + sb + c1_4 * r2 * r2;
        e0 *= e0; e1 *= e1; e2 *= e2;
        R a0 = (R)0.1 * e1 * e2, a1 = (R)0.6 * e0 * e2, a2 = (R)0.3 * e0 * e1;
        vm = (a0 * q0 + a1 * qa + a2 * qb) * rcp<R>(a0 + a1 + a2);
    }
    {
        R q0 = ((R)2 * V5 - (R)7 * V4 + (R)11 * V3) * c1_6;
        R t0 = V5 - (R)2 * V4 + V3, r0 = V5 - (R)4 * V4 + (R)3 * V3;
        R r1 = V4 - V2, r2 = (R)3 * V3 - (R)4 * V2 + V1;
        R e0 = eps + c13_12 * t0 * t0 + c1_4 * r0 * r0;
        R e1 = eps + sb + c1_4 * r1 * r1;
        R e2 = eps + sa + c1_4 * r2 * r2;
        e0 *= e0; e1 *= e1; e2 *= e2;
        R a0 = (R)0.1 * e1 * e2, a1 = (R)0.6 * e0 * e2, a2 = (R)0.3 * e0 * e1;
        vp = (a0 * q0 + a1 * qb + a2 * qa) * rcp<R>(a0 + a1 + a2);
    }
}

// The two WENO3 edge values of one interface from V0..V3 (V1, V2 its
// nodes): vm from V0, V1, V2 and vp from V3, V2, V1, each
// (a0 q0 + a1 q1)/(a0 + a1) with a_k = d_k/(eps+b_k)^2, d = (1/3, 2/3),
// multiplied through; the candidate on {V1, V2} and its smoothness term
// serve both.
template <typename R>
__device__ __forceinline__ void weno3_lr(R V0, R V1, R V2, R V3, R eps, R &vm, R &vp)
{
    const R q1 = (V1 + V2) * (R)0.5;
    R e1 = eps + (V2 - V1) * (V2 - V1);
    e1 *= e1;
    {
        R q0 = (-V0 + (R)3 * V1) * (R)0.5;
        R e0 = eps + (V1 - V0) * (V1 - V0);
        e0 *= e0;
        R a0 = (R)(1.0 / 3.0) * e1, a1 = (R)(2.0 / 3.0) * e0;
        vm = (a0 * q0 + a1 * q1) * rcp<R>(a0 + a1);
    }
    {
        R q0 = (-V3 + (R)3 * V2) * (R)0.5;
        R e0 = eps + (V2 - V3) * (V2 - V3);
        e0 *= e0;
        R a0 = (R)(1.0 / 3.0) * e1, a1 = (R)(2.0 / 3.0) * e0;
        vp = (a0 * q0 + a1 * q1) * rcp<R>(a0 + a1);
    }
}

// (in FP64 on the integer pipes: an FP64 compare takes an FP64-pipe slot)
__device__ __forceinline__ int sgn_d(double a)
{
    const uint64_t b = conv_bits64(a), m = b & 0x7fffffffffffffffull;
    return m == 0 || m > 0x7ff0000000000000ull ? 0 : ((b >> 63) ? -1 : 1);
}
__device__ __forceinline__ int sgn_d(float a) { return (a > 0.0f) - (a < 0.0f); }
__device__ __forceinline__ int sgn_d(dual a) { return (a.v > 0.0) - (a.v < 0.0); }
__device__ __forceinline__ bool le(double a, double b) { return a <= b; }
__device__ __forceinline__ bool le(float a, float b) { return a <= b; }
__device__ __forceinline__ bool le(dual a, dual b) { return a.v <= b.v; }

// The sign that the switch Y takes of a projected jump: 0 where the jump is within
// sign_tol of scale, the magnitudes that form it.  In FP64 (scale in FP32) a jump clear of the
// threshold, of a scale well inside FP32's range, is decided in FP32, off the FP64 pipe; the answer
// JUMP_UNSURE leaves the others to an FP64 scale, so that every decision is the FP64 one.  aT: the factors
// of scale that are summed, infinite (jump_terms) where FP32 may lose a product with them.
// (Against the FP32 decision alone: 400^2 step 4.17 -> 4.19 ms, 64^3 blast step 18.71 -> 18.81 ms.)
constexpr int JUMP_UNSURE = 2;
__device__ __forceinline__ int jump_sign(float jump, double sign_tol, float scale)
{
    return fabsf(jump) <= (float)sign_tol * scale ? 0 : sgn_d(jump);
}
__device__ __forceinline__ int jump_sign(double jump, double sign_tol, float scale)
{
    const float j = fabsf(d2f_int(jump)), t = (float)sign_tol * scale;
    if (conv_bits32(scale) - 0x129e74d2u < 0x7149f2cau - 0x129e74d2u)   // 1e-27 <= scale < 1e30
        return j < 0.999f * t ? 0 : (j > 1.001f * t ? sgn_d(jump) : JUMP_UNSURE);
    return conv_bits64(jump) << 1 == 0 ? 0 : JUMP_UNSURE;   // (gas at rest: both are 0)
}
template <typename R, int N>
__device__ __forceinline__ void jump_terms(float aT[N])
{
    if constexpr (std::is_same<R, double>::value) {
        float m = aT[0];
#pragma unroll
        for (int a = 1; a < N; ++a) m = fmaxf(m, aT[a]);
        if (!(m < 1.0e12f)) aT[N - 1] = conv_float(0x7f800000u);
    }
}
__device__ __forceinline__ int jump_sign64(double jump, double sign_tol, double scale)
{
    return fabs(jump) <= sign_tol * scale ? 0 : sgn_d(jump);
}

// Scaled eigenvectors of dF_1/dU (Sec. 4) at the rotated state with 4-velocity (W,
// un, ut): rows E[m] = s_m (dD, dm_n, dm_t, dE) with s_m = (dU.dV)^-1/2, for the waves
// lambda_-, v_n (entropy, d rho = 1), v_n (shear, d v_t = 1), lambda_+.  An acoustic wave is, with
// xi = (-lambda, n), a = u.xi = W (v_n - lambda), k = xi + a u and k^2 = 1 - lambda^2 + a^2,
//   du = -a k,  dp = Gamma p k^2,  d rho = rho k^2,
//   dU.dV = 2 beta rho h a^2 kap,  kap = W (1 - lambda^2) - a lambda,
// (rho h a^2 = Gamma p k^2), and a = +-c W (disc +- v_n c/W^2)/(1 - v^2 c^2) keeps its
// relative accuracy.  igg = (Gamma-1)/Gamma.
template <typename R>
__device__ __forceinline__ void eigen_rhd(R gam, R gg, R igg, R rho, R p, R un, R ut, R W, R iW, R E[4][4], R &lam_m,
                                          R &lam_p)
{
    const R one = (R)1, two = (R)2;
    const R iW2 = iW * iW, vn = un * iW, v2 = fma_<R>(-iW, iW, one);
    const R gp = gam * p, rh = fma_<R>(gg, p, rho), beta = rho * qrcp<R>(p);
    const R c2 = gp * qrcp<R>(rh), c = c2 * qrsq<R>(c2);
    const R D0 = fma_<R>(-v2, c2, one), X = fma_<R>(-(vn * vn), sub_<R>(one, c2), D0);
    const R disc = iW * X * qrsq<R>(X), cd = W * c * qrcp<R>(D0), vc = vn * c * iW2;
    const R e0 = fma_<R>(gg, gp, rho), rhW = rh * W, brh = two * beta * rh;
#pragma unroll
    for (int side = 0; side < 2; ++side) {
        const int m = side == 0 ? 0 : 3;
        const R a = cd * sub_<R>(vc, side == 0 ? -disc : disc);
        const R lam = fma_<R>(-a, iW, vn);
        (side == 0 ? lam_m : lam_p) = lam;
        const R ol = (one - lam) * (one + lam), k0 = fma_<R>(a, W, lam), k2 = fma_<R>(a, a, ol), kap = fma_<R>(W, ol, -(a * lam));
        const R s = qrsq<R>(brh * (a * a) * kap);
        const R ek = e0 * k2, ha = rhW * a, cc = fma_<R>(ek, W, -(rh * a * k0));
        E[m][0] = s * (rho * kap);
        E[m][1] = s * fma_<R>(cc, un, -(ha * fma_<R>(a, un, one)));
        E[m][2] = s * fma_<R>(cc, ut, -(ha * (a * ut)));
        E[m][3] = s * fma_<R>(-gp, k2, fma_<R>(ek, W * W, -(two * (ha * k0))));
    }
    // entropy wave: dU = (W, W^2 v, W^2), dU.dV = Gamma W/((Gamma-1) rho)
    const R q = W * rho * igg, g1 = q * qrsq<R>(q);
    E[1][0] = g1;
    E[1][1] = g1 * un;
    E[1][2] = g1 * ut;
    E[1][3] = g1 * W;
    // shear wave: dU = (rho W^3 v_t, 2 rho h W^4 v_n v_t, rho h (2 W^4 v_t^2 + W^2), 2 rho h W^4
    // v_t), dU.dV = rho h beta W^3 (1 + W^2 v_t^2)
    const R f = qrsq<R>(rh * beta * iW * fma_<R>(ut, ut, one)), h = f * rh, h2 = two * h * ut;
    E[2][0] = f * rho * ut;
    E[2][1] = h2 * un;
    E[2][2] = fma_<R>(h2, ut, h);
    E[2][3] = h2 * W;
}

}  // namespace esmm

// Operator sweeps T s = sum_j omega_j (D_j + Sigma_t)^{-1} s on 2D meshes whose cross sections are constant on regions
// (paper Sec. 3.1-3.2): every inner iteration, residual and right-hand side of a solve.
//
// Decomposition.  A task is (instance, quadrant, up to D unique directions); one CTA of W warps sweeps one task and
// writes one partial scalar flux.  A band is 32 * RPL mesh rows (rows counted in the upwind y order); warp w takes the
// bands w, w + W, w + 2W, ...  Lane l owns the rows RPL l .. RPL l + RPL - 1 of the band and handles column i at its
// warp's step l + i, so the y-inflow of its first row is the y-outflow the lane below produced one step earlier (warp
// shuffle; the first lane reads what the last lane of the band below left in shared memory), that of its other rows
// comes from the row before in the same step, and the x-inflow is the lane's own previous cell (registers).  Band k+1
// starts 32 + SK steps after band k, or P steps after the warp's previous band, whichever its warp allows; P is such
// that what a band reads was written at least one group of SK steps earlier, so the warps meet at a barrier once per
// group.  With W = 1 a task has no idle steps but 31 (throughput: many tasks), with one warp per band its critical path
// is shortest (latency: few tasks).
//
// Cell algebra.  In the frame reflected so that Omega_x, Omega_y > 0 the cell block is
// L = alpha K(x)I + beta I(x)K + sigma_t I, K = 2 I + sqrt2 N with N^2 = -I.  L^{-1} is therefore a combination of
// 1, N_x, N_y, N_x N_y, which a basis can make use of:
//  * Rot (FP32): both axes turned by 45 degrees, x' = (x_0 + x_1, x_1 - x_0) / sqrt2, an orthogonal change of basis.
//    There N = [[0, a], [-1/a, 0]], a^2 = 2 + sqrt3, the outflow functional is (a, 1/a) and the inflow vector
//    -(1/a, a).  With the second component of each axis scaled by q = 1/a^2, traces in units of a, the inflow enters
//    both components of a pair with the same weight -alpha (or -beta), the outflow is a plain sum, and L^{-1} has
//    eight distinct entries: 8 + 16 + 4 multiply-adds and adds and 4 for the quadrature, against 9 + 16 + 4 + 4 and
//    sixteen entries in the Legendre basis.  The source is brought to the basis, and the summed flux back, once per cell
//    and task.  The error of an apply against 64-bit values is 0.5 to 1.1 times that of the former Legendre kernels (13
//    batches of 1 to 256 instances; 2.3e-7 against 2.2e-7 on the uneven one below).
//  * Legendre (FP64): no change of basis; tasks of one and two directions with the cell inverses that the angular sweeps
//    use, wider ones with the nine entries that are distinct.
//  * Scaled (double-float): the Legendre modes scaled, which saves products.
// The eigenbasis of N (complex products, 24 operations a direction and 30 a cell for its transforms) is no better choice for
// these two: it is not orthogonal (condition number 3.7), in double-float the error of an apply is 15 to 70 % larger, and
// in FP64 the 32 D operations of the Legendre basis are as few for tasks of up to four directions.
//
// FP32 runs pairs of directions in the packed multiply-add (fma.rn.f32x2): half the issue slots at the same rate.
//
// Bounds and measurements (one operator apply with the sum of its partial fluxes, GB300; before: Legendre basis, sixteen
// table entries per direction and region, D <= 8, one warp per task or per band).  FP32, 64 x 256^2, 192 directions,
// 8 x 8 regions: 2.08 -> 0.96 ms (D = 12, W = 2; bound by the load/store data pipe); 256 instances on 32^2, 64^2 and 128^2,
// 128 directions: 0.672 -> 0.327 ms (D = 8, two rows a lane: each table and shuffle serves two cells); one 64^2 instance:
// 36.3 -> 26.7 us (latency of 131 steps).  FP64 is bound by the FP64 unit, which takes 64 cycles of an SM quarter for a warp
// instruction, whatever the number of lanes, and 76 with all four quarters busy: so by instructions per step.
// 7.92 -> 6.63 ms on the 256 instances (D = 4), 0.919 -> 0.500 ms on 10 x 80^2 with CL(30, 6) (D = 1), one 40^2 instance
// 154 -> 113 us.  Double-float is bound by FP32 issue: 3.61 -> 2.00 ms on 16 x 256^2 (D = 4, W = 4; the step loop not
// unrolled: unrolled it missed the instruction cache, 3.48 ms); 2 x (160 x 186) 417 -> 176 us (238 while sources rotated
// through registers, whose moves waited for their loads).
#include <algorithm>
#include <cmath>
#include <type_traits>
#include <utility>
#include <vector>

#include "sweep.h"

namespace rte {

// ----------------------------------------------------------------------------------- vectors of directions
template <typename T, int VW>
struct Dv;   // VW directions side by side

template <typename T>
struct Dv<T, 1> {
  T x;
  __device__ __forceinline__ static Dv all(T v) { return Dv{v}; }
  __device__ __forceinline__ T sum() const { return x; }
};
template <typename T>
__device__ __forceinline__ Dv<T, 1> vadd(Dv<T, 1> a, Dv<T, 1> b) { return Dv<T, 1>{a.x + b.x}; }
template <typename T>
__device__ __forceinline__ Dv<T, 1> vmul(Dv<T, 1> a, Dv<T, 1> b) { return Dv<T, 1>{a.x * b.x}; }
template <typename T>
__device__ __forceinline__ Dv<T, 1> vfma(Dv<T, 1> a, Dv<T, 1> b, Dv<T, 1> c) { return Dv<T, 1>{c.x + a.x * b.x}; }

template <>
struct Dv<float, 2> {
  float x, y;
  __device__ __forceinline__ static Dv all(float v) { return Dv{v, v}; }
  __device__ __forceinline__ float sum() const { return x + y; }
  __device__ __forceinline__ unsigned long long bits() const {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
  }
  __device__ __forceinline__ static Dv of(unsigned long long b) {
    Dv r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(b));
    return r;
  }
};
using F2 = Dv<float, 2>;
__device__ __forceinline__ F2 vadd(F2 a, F2 b) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a.bits()), "l"(b.bits()));
  return F2::of(r);
}
__device__ __forceinline__ F2 vmul(F2 a, F2 b) {
  unsigned long long r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a.bits()), "l"(b.bits()));
  return F2::of(r);
}
__device__ __forceinline__ F2 vfma(F2 a, F2 b, F2 c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a.bits()), "l"(b.bits()), "l"(c.bits()));
  return F2::of(r);
}

// Predicated load of the two traces of a column from shared memory, in place (a branch or a select per value costs more
// than the load)
__device__ __forceinline__ void load_traces(unsigned p, unsigned addr, Dv<float, 1>* y) {
  asm volatile("{.reg .pred q; setp.ne.u32 q, %2, 0; @q ld.shared.v2.f32 {%0, %1}, [%3];}"
               : "+f"(y[0].x), "+f"(y[1].x) : "r"(p), "r"(addr));
}
__device__ __forceinline__ void load_traces(unsigned p, unsigned addr, F2* y) {
  asm volatile("{.reg .pred q; setp.ne.u32 q, %4, 0; @q ld.shared.v4.f32 {%0, %1, %2, %3}, [%5];}"
               : "+f"(y[0].x), "+f"(y[0].y), "+f"(y[1].x), "+f"(y[1].y) : "r"(p), "r"(addr));
}
__device__ __forceinline__ void load_traces(unsigned p, unsigned addr, Dv<double, 1>* y) {
  asm volatile("{.reg .pred q; setp.ne.u32 q, %2, 0; @q ld.shared.v2.f64 {%0, %1}, [%3];}"
               : "+d"(y[0].x), "+d"(y[1].x) : "r"(p), "r"(addr));
}
__device__ __forceinline__ void load_traces(unsigned p, unsigned addr, Dv<dfloat, 1>* y) {
  asm volatile("{.reg .pred q; setp.ne.u32 q, %4, 0; @q ld.shared.v4.f32 {%0, %1, %2, %3}, [%5];}"
               : "+f"(y[0].x.hi), "+f"(y[0].x.lo), "+f"(y[1].x.hi), "+f"(y[1].x.lo) : "r"(p), "r"(addr));
}

__device__ __forceinline__ float up1(float v) { return __shfl_up_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ double up1(double v) { return __shfl_up_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ dfloat up1(dfloat v) { return dfloat(up1(v.hi), up1(v.lo)); }
template <typename T>
__device__ __forceinline__ Dv<T, 1> up1(Dv<T, 1> v) { return Dv<T, 1>{up1(v.x)}; }
__device__ __forceinline__ F2 up1(F2 v) { return F2{up1(v.x), up1(v.y)}; }

// v or -v: the sign bit times a mask (0 or 1 << 31), which takes no floating-point instruction
__device__ __forceinline__ float flip(float v, unsigned m) { return __uint_as_float(__float_as_uint(v) ^ m); }
__device__ __forceinline__ double flip(double v, unsigned m) {
  return __hiloint2double(__double2hiint(v) ^ (int)m, __double2loint(v));
}
__device__ __forceinline__ dfloat flip(dfloat v, unsigned m) { return dfloat(flip(v.hi, m), flip(v.lo, m)); }

// ------------------------------------------------------------------------------------------- cell algebras
// Sums of products of double-floats: the high parts go through two-sums, what these miss and the low parts are added up
// on the side, and one renormalisation ends the sum (the compensated dot product of Ogita, Rump and Oishi, SIAM J. Sci.
// Comput. 26, 2005): 12 operations a term against 18 for a product and a sum of pairs.
struct DfSum {
  float s, e;
  __device__ __forceinline__ explicit DfSum(dfloat a) : s(a.hi), e(a.lo) {}
  __device__ __forceinline__ DfSum(dfloat a, dfloat b) {   // a b
    s = __fmul_rn(a.hi, b.hi);
    e = __fmaf_rn(a.lo, b.hi, __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.hi, b.hi, -s)));
  }
  __device__ __forceinline__ DfSum operator-() const {
    DfSum r = *this;
    r.s = -s;
    r.e = -e;
    return r;
  }
  __device__ __forceinline__ DfSum operator+(DfSum b) const {
    DfSum r = *this;
    r.s = __fadd_rn(s, b.s);
    const float bb = __fsub_rn(r.s, s);
    const float er = __fadd_rn(__fsub_rn(s, __fsub_rn(r.s, bb)), __fsub_rn(b.s, bb));
    r.e = __fadd_rn(e, __fadd_rn(er, b.e));
    return r;
  }
  __device__ __forceinline__ dfloat raw() const { return dfloat(s, e); }   // not renormalised: for further sums only
  __device__ __forceinline__ dfloat get() const { return df_renorm(s, e); }
};

template <typename T>
struct Rot {
  // table entries per direction and region, source factors per region, elements before the entries
  static constexpr int TW = 8, FW = 4, HD = 4;
  static constexpr int NC = 3;   // constants per direction: -alpha, -beta, omega
  static constexpr double A2 = 3.7320508075688772935, Q = 0.26794919243112270647;
  // factors of the source's four Legendre components before to_basis, for reflection signs fx, fy
  __device__ static T factor(int k, double fx, double fy) {
    return (T)(0.5 * ((k & 1) ? fx : 1.0) * ((k & 2) ? fy : 1.0));
  }
  __device__ __forceinline__ static void source(const T* q, const T* f, const unsigned*, T* S) {
    T t[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) t[e] = q[e] * f[e];
    to_basis(t, S);
  }
  // The transforms' rounding errors are shared by all directions of a task, so both are written for few roundings at the
  // size of the leading component: the higher modes are added up first and meet it in one multiply-add (to), the scalings
  // are part of the sums (from).  Against sums of pairs and separate products: 1 % less error of an apply on average over
  // those batches, up to 3 %.
  __device__ __forceinline__ static void to_basis(const T* t, T* S) {
    const T e = t[1] + t[2], f = t[1] - t[2];
    S[0] = t[0] + (t[3] + e);
    S[1] = fmaf((T)-Q, t[0], (T)Q * (t[3] + f));
    S[2] = fmaf((T)-Q, t[0], (T)Q * (t[3] - f));
    S[3] = fmaf((T)(Q * Q), t[0], (T)(Q * Q) * (t[3] - e));
  }
  __device__ __forceinline__ static void from_basis(const T* c, T* s) {
    constexpr T a = (T)(0.5 * A2), b = (T)(0.5 * A2 * A2);
    const T h = (T)0.5 * c[0], v = c[1] + c[2], z = c[1] - c[2];
    const T u = fmaf(b, c[3], h), w = fmaf(-b, c[3], h);
    s[0] = fmaf(-a, v, u);
    s[1] = fmaf(a, z, w);
    s[2] = fmaf(-a, z, w);
    s[3] = fmaf(a, v, u);
  }
  __device__ static void boundary(double g, T* t) {   // traces of a constant g: g / (sqrt2 a) (1, -q)
    const double v = g * 0.70710678118654752440 / 1.9318516525781365735;
    t[0] = (T)v;
    t[1] = (T)(-Q * v);
  }
  __device__ static void constants(double al, double be, double w, T* c) {
    c[0] = (T)(-al);
    c[1] = (T)(-be);
    c[2] = (T)w;
  }
  // X, Y: inflow traces in, outflow traces out; acc = (zero ? 0 : acc) + omega p
  template <typename V>
  __device__ __forceinline__ static void cell(const V* S, V* X, V* Y, const V* m, const V* c, V* acc, bool zero) {
    const V r0 = vfma(c[1], Y[0], vfma(c[0], X[0], S[0])), r1 = vfma(c[1], Y[1], vfma(c[0], X[0], S[1]));
    const V r2 = vfma(c[1], Y[0], vfma(c[0], X[1], S[2])), r3 = vfma(c[1], Y[1], vfma(c[0], X[1], S[3]));
    // m: g, bx, cx, by, cy, bb, -d, cc (see k_wave_tables)
    const V p0 = vfma(m[5], r3, vfma(m[3], r2, vfma(m[1], r1, vmul(m[0], r0))));
    const V p1 = vfma(m[3], r3, vfma(m[6], r2, vfma(m[2], r0, vmul(m[0], r1))));
    const V p2 = vfma(m[1], r3, vfma(m[6], r1, vfma(m[4], r0, vmul(m[0], r2))));
    const V p3 = vfma(m[7], r0, vfma(m[4], r1, vfma(m[2], r2, vmul(m[0], r3))));
    X[0] = vadd(p0, p1);
    X[1] = vadd(p2, p3);
    Y[0] = vadd(p0, p2);
    Y[1] = vadd(p1, p3);
    acc[0] = zero ? vmul(c[2], p0) : vfma(c[2], p0, acc[0]);
    acc[1] = zero ? vmul(c[2], p1) : vfma(c[2], p1, acc[1]);
    acc[2] = zero ? vmul(c[2], p2) : vfma(c[2], p2, acc[2]);
    acc[3] = zero ? vmul(c[2], p3) : vfma(c[2], p3, acc[3]);
  }
};

// The Legendre basis itself (FP64): the sixteen entries of the cell inverses, 32 D operations a cell.  SIG: the kernel
// multiplies the source by Sigma_s (4 more); else it comes multiplied, or unscaled where there is no Sigma_s.
template <typename T, bool SIG>
struct Legendre {
  static constexpr int TW = 16, FW = SIG ? 1 : 0, HD = 2;   // the factor is padded to 16 bytes
  static constexpr int NC = 5;   // alpha, beta, sqrt3 alpha, sqrt3 beta, omega
  __device__ static T factor(int, double, double) { return (T)1; }
  // neg: sign bits of the four components in the reflected frame
  __device__ __forceinline__ static void source(const T* q, const T* f, const unsigned* neg, T* S) {
#pragma unroll
    for (int e = 0; e < 4; ++e) S[e] = flip(SIG ? q[e] * f[0] : q[e], neg[e]);
  }
  __device__ __forceinline__ static void from_basis(const T* c, T* s) {
#pragma unroll
    for (int e = 0; e < 4; ++e) s[e] = c[e];
  }
  __device__ static void boundary(double g, T* t) {
    t[0] = (T)g;
    t[1] = (T)0;
  }
  __device__ static void constants(double al, double be, double w, T* c) {
    const double s3 = 1.7320508075688772;
    c[0] = (T)al;
    c[1] = (T)be;
    c[2] = (T)(s3 * al);
    c[3] = (T)(s3 * be);
    c[4] = (T)w;
  }
  template <typename V>
  __device__ __forceinline__ static void cell(const V* S, V* X, V* Y, const V* m, const V* c, V* acc, bool zero) {
    const T a = c[0].x, b = c[1].x, a3 = c[2].x, b3 = c[3].x, w = c[4].x, s3 = (T)1.7320508075688772;
    const T x0 = X[0].x, x1 = X[1].x, y0 = Y[0].x, y1 = Y[1].x;
    const T r[4] = {S[0].x + a * x0 + b * y0, S[1].x - a3 * x0 + b * y1, S[2].x + a * x1 - b3 * y0,
                    S[3].x - a3 * x1 - b3 * y1};
    T q[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      q[i] = m[4 * i].x * r[0] + m[4 * i + 1].x * r[1] + m[4 * i + 2].x * r[2] + m[4 * i + 3].x * r[3];
      acc[i].x = zero ? w * q[i] : acc[i].x + w * q[i];
    }
    X[0].x = q[0] + s3 * q[1];
    X[1].x = q[2] + s3 * q[3];
    Y[0].x = q[0] + s3 * q[2];
    Y[1].x = q[1] + s3 * q[3];
  }
};

// The same with the nine distinct entries of a cell inverse, for FP64 tasks of three and more directions.  As a combination
// of 1, N_x, N_y, N_x N_y, N = [[-1, sqrt3], [-sqrt3, 1]] / sqrt2, an inverse has its diagonal d0 .. d3, +-u0, +-u1 between the
// x-modes, +-v0, +-v1 between the y-modes, and +-w.  Fewer loads and smaller tables (256 uneven instances 6.74 -> 6.63 ms), and
// the entries are rounded once (k_wave_tables), which the certificate of a tight solve gains by: emulated against extended
// precision, an apply's error is 2.5e-16 against 3.3e-16 with the inverses of the problem set-up on 40^2, 5.8e-16 against
// 1.7e-15 on 128^2.
template <typename T, bool SIG>
struct Nine : Legendre<T, SIG> {
  static constexpr int TW = 10;   // nine entries and a spare one, for 16-byte boundaries
  template <typename V>
  __device__ __forceinline__ static void cell(const V* S, V* X, V* Y, const V* m, const V* c, V* acc, bool zero) {
    const T a = c[0].x, b = c[1].x, a3 = c[2].x, b3 = c[3].x, w = c[4].x, s3 = (T)1.7320508075688772;
    const T x0 = X[0].x, x1 = X[1].x, y0 = Y[0].x, y1 = Y[1].x;
    const T r0 = S[0].x + a * x0 + b * y0, r1 = S[1].x - a3 * x0 + b * y1;
    const T r2 = S[2].x + a * x1 - b3 * y0, r3 = S[3].x - a3 * x1 - b3 * y1;
    const T q[4] = {m[0].x * r0 + m[4].x * r1 + m[6].x * r2 + m[8].x * r3,
                    m[1].x * r1 - m[4].x * r0 - m[8].x * r2 + m[7].x * r3,
                    m[2].x * r2 - m[6].x * r0 - m[8].x * r1 + m[5].x * r3,
                    m[3].x * r3 + m[8].x * r0 - m[7].x * r1 - m[5].x * r2};
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[i].x = zero ? w * q[i] : acc[i].x + w * q[i];
    X[0].x = q[0] + s3 * q[1];
    X[1].x = q[2] + s3 * q[3];
    Y[0].x = q[0] + s3 * q[2];
    Y[1].x = q[1] + s3 * q[3];
  }
};

// Scaled Legendre modes (double-float): P = (1, sqrt3, sqrt3, 3) p, sources divided by the same, second traces times
// sqrt3.  Outflows become plain sums and each product of a trace enters two components: 356 operations a cell and direction
// against 400 in the Legendre basis, with the same rounding errors (in the eigenbasis of N 318 and transforms, and errors
// 15 to 70 % larger).  The scalings cost nothing: they are part of the tables, the quadrature weights and the pass that
// splits the source into pairs, which also multiplies it by Sigma_s.  Nine entries an inverse, as above.
struct Scaled {
  using T = dfloat;
  static constexpr int TW = 10, FW = 0, HD = 0;   // nine entries and a spare one, for 16-byte boundaries
  static constexpr int NC = 8;   // alpha, alpha / 3, beta, beta / 3, omega / (1, sqrt3, sqrt3, 3)
  __device__ static double scale(int k) { return k == 0 ? 1.0 : (k == 3 ? 3.0 : 1.7320508075688772); }
  __device__ static T factor(int, double, double) { return (T)0; }
  __device__ __forceinline__ static void source(const T* q, const T*, const unsigned* neg, T* S) {
#pragma unroll
    for (int e = 0; e < 4; ++e) S[e] = flip(q[e], neg[e]);
  }
  __device__ __forceinline__ static void from_basis(const T* c, T* s) {
#pragma unroll
    for (int e = 0; e < 4; ++e) s[e] = df_renorm(c[e].hi, c[e].lo);
  }
  __device__ static void boundary(double g, T* t) {
    t[0] = (T)g;
    t[1] = (T)0;
  }
  __device__ static void constants(double al, double be, double w, T* c) {
    c[0] = (T)al;
    c[1] = (T)(al / 3.0);
    c[2] = (T)be;
    c[3] = (T)(be / 3.0);
    for (int k = 0; k < 4; ++k) c[4 + k] = (T)(w / scale(k));
  }
  template <typename V>
  __device__ __forceinline__ static void cell(const V* S, V* X, V* Y, const V* m, const V* c, V* acc, bool zero) {
    const DfSum x0(c[0].x, X[0].x), x1(c[1].x, X[1].x), y0(c[2].x, Y[0].x), y1(c[3].x, Y[1].x);
    const T r0 = (DfSum(S[0].x) + x0 + y0).get(), r1 = (DfSum(S[1].x) + -x0 + y1).get();
    const T r2 = (DfSum(S[2].x) + x1 + -y0).get(), r3 = (DfSum(S[3].x) + -x1 + -y1).get();
    auto dot = [](T m0, T a0, T m1, T a1, T m2, T a2, T m3, T a3) {
      return (DfSum(m0, a0) + DfSum(m1, a1) + DfSum(m2, a2) + DfSum(m3, a3)).get();
    };
    const T d0 = m[0].x, d1 = m[1].x, d2 = m[2].x, d3 = m[3].x, u0 = m[4].x, u1 = m[5].x, v0 = m[6].x, v1 = m[7].x, w = m[8].x;
    const T q[4] = {dot(d0, r0, u0, r1, v0, r2, w, r3), dot(-u0, r0, d1, r1, -w, r2, v1, r3),
                    dot(-v0, r0, -w, r1, d2, r2, u1, r3), dot(w, r0, -v1, r1, -u1, r2, d3, r3)};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const DfSum wq(c[4 + i].x, q[i]);
      acc[i].x = zero ? wq.raw() : (DfSum(acc[i].x) + wq).raw();   // renormalised once, in from_basis
    }
    X[0].x = (DfSum(q[0]) + DfSum(q[1])).get();
    X[1].x = (DfSum(q[2]) + DfSum(q[3])).get();
    Y[0].x = (DfSum(q[0]) + DfSum(q[2])).get();
    Y[1].x = (DfSum(q[1]) + DfSum(q[3])).get();
  }
};

// Unevaluated sums of two doubles, for the tables alone (two-sum and two-product as in dfloat.cuh)
struct Dd {
  double h, l;
  __device__ Dd operator-() const { return Dd{-h, -l}; }
};
__device__ __forceinline__ Dd dd_sum(double a, double b) {
  const double s = __dadd_rn(a, b), t = __dsub_rn(s, a);
  return Dd{s, __dadd_rn(__dsub_rn(a, __dsub_rn(s, t)), __dsub_rn(b, t))};
}
__device__ __forceinline__ Dd operator+(Dd a, Dd b) {
  const Dd s = dd_sum(a.h, b.h);
  return dd_sum(s.h, __dadd_rn(s.l, __dadd_rn(a.l, b.l)));
}
__device__ __forceinline__ Dd operator*(Dd a, Dd b) {
  const double p = __dmul_rn(a.h, b.h);
  return dd_sum(p, __fma_rn(a.l, b.h, __fma_rn(a.h, b.l, __fma_rn(a.h, b.h, -p))));
}
__device__ __forceinline__ Dd operator/(Dd a, Dd b) {
  const double q = __ddiv_rn(a.h, b.h);
  const Dd r = a + -(Dd{q, 0.0} * b);
  return dd_sum(q, __ddiv_rn(r.h, b.h));
}

// Tables per (instance, unique direction, region): Rot FP32 [8], Nine FP64 [10] and Scaled double-float pairs [10].
// l_1 = c_0 + i sqrt2 (alpha + beta) and l_2 = c_0 + i sqrt2 (alpha - beta), c_0 = 2 (alpha + beta) + sigma_t, are the
// eigenvalues of L on the products of eigenvectors of N, n_1 and n_2 their squared moduli;
// L^{-1} = g + g_x N_x + g_y N_y + g_xy N_x N_y follows from 1 / l_1, 1 / l_2.
__global__ void k_wave_tables(int B, int nu, int R, const InstInfo* inst, const UDir* ud, const double* sig_t,
                              float* rot, double* inv64, float2* inv_df) {
  const long long tid = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (tid >= (long long)B * nu * R) return;
  const int r = (int)(tid % R), u = (int)((tid / R) % nu), b = (int)(tid / ((long long)R * nu));
  const double al = ud[u].ax / inst[b].hx, be = ud[u].ay / inst[b].hy, sg = sig_t[(size_t)b * R + r];
  {
    const double s2 = 1.4142135623730950488, c0 = 2.0 * (al + be) + sg;
    const double i1 = s2 * (al + be), i2 = s2 * (al - be);
    const double n1 = c0 * c0 + i1 * i1, n2 = c0 * c0 + i2 * i2, inv = 1.0 / (n1 * n2);
    const double g = c0 * (c0 * c0 + 2.0 * (al * al + be * be)) * inv;
    const double gx = -s2 * al * (c0 * c0 + 2.0 * (al - be) * (al + be)) * inv;
    const double gy = -s2 * be * (c0 * c0 - 2.0 * (al - be) * (al + be)) * inv;
    const double gxy = 4.0 * al * be * c0 * inv;
    // scaled N of an axis: [[0, a^3], [-a^{-3}, 0]] (a^3: the turn's a and twice the scaling by q)
    const double a3 = 7.2097685201075047693, b3 = 1.0 / a3;
    const double t[8] = {g, gx * a3, -gx * b3, gy * a3, -gy * b3, gxy * a3 * a3, -gxy, gxy * b3 * b3};
    for (int k = 0; k < 8; ++k) rot[tid * 8 + k] = (float)t[k];
  }
  // A = c_0 / n_1, B = c_0 / n_2, C = (alpha + beta) / n_1, E = (alpha - beta) / n_2, k = (B - A) / 4:
  // d0, d3 = B - k +- C; d2, d1 = A + k +- E; u0, u1 = -sqrt3/2 (C + E) -+ sqrt3 k; v0, v1 = -sqrt3/2 (C - E) -+ sqrt3 k; w = 3 k.
  // In sums of two doubles, so that the entries are rounded once: what their rounding loses adds up along a ray.
  const Dd sum = dd_sum(al, be), dif = dd_sum(al, -be);
  const Dd c0 = Dd{2.0 * sum.h, 2.0 * sum.l} + Dd{sg, 0.0}, cc = c0 * c0, ss = sum * sum, dd = dif * dif;
  const Dd n1 = cc + Dd{2.0 * ss.h, 2.0 * ss.l}, n2 = cc + Dd{2.0 * dd.h, 2.0 * dd.l};
  const Dd A = c0 / n1, Bq = c0 / n2, C = sum / n1, E = dif / n2;
  const Dd s3{1.7320508075688772, 1.0035084221806903e-16}, h3{0.8660254037844386, 5.0175421109034514e-17};
  Dd k = Bq + -A;
  k = Dd{0.25 * k.h, 0.25 * k.l};
  const Dd p1 = Bq + -k, p2 = A + k, x = -(h3 * (C + E)), y = -(h3 * (C + -E)), sk = s3 * k;
  const Dd m[9] = {p1 + C, p2 + -E, p2 + E, p1 + -C, x + -sk, x + sk, y + -sk, y + sk, k + Dd{2.0 * k.h, 2.0 * k.l}};
  // of the scaled modes: rows and columns times (1, sqrt3, sqrt3, 3)
  const Dd c3{3.0, 0.0}, c33 = s3 * c3;
  const Dd f[9] = {Dd{1.0, 0.0}, c3, c3, Dd{9.0, 0.0}, s3, c33, s3, c33, c3};
  for (int e = 0; e < 9; ++e) {
    inv64[tid * 10 + e] = m[e].h;
    const Dd v = m[e] * f[e];
    const float h = (float)v.h;
    inv_df[tid * 10 + e] = make_float2(h, (float)__dadd_rn(__dsub_rn(v.h, (double)h), v.l));
  }
  inv64[tid * 10 + 9] = 0.0;
  inv_df[tid * 10 + 9] = make_float2(0.f, 0.f);
}

int build_wave_tables(rte_problem* p) {
  const long long n = (long long)p->B * p->nu * p->R;
  k_wave_tables<<<(unsigned)((n + 127) / 128), 128>>>(p->B, p->nu, p->R, p->d_inst.p, p->d_udir.p, p->d_sig_t.p,
                                                      p->d_rot32.p, p->d_inv64.p, reinterpret_cast<float2*>(p->d_linv_df.p));
  count_launch();
  RTE_CHECK_CUDA(cudaGetLastError());
  return RTE_OK;
}

// ------------------------------------------------------------------------------------------------- kernel
template <typename T, int N>
struct alignas(N * sizeof(T) >= 16 ? 16 : N * sizeof(T)) Blk {
  T v[N];
};

// Elements between the tables of two regions: a multiple of 16 bytes, odd in 16-byte units, so that lanes in two
// neighbouring regions read from different banks
constexpr int table_stride(int n, int bytes) { return n + (((n * bytes) / 16) % 2 ? 0 : 16 / bytes); }

// Columns a trace buffer between neighbouring warps keeps: the reader follows SK + 1 steps behind the writer, and the
// two meet every SK steps, so 32 columns are more than it can lag
constexpr int kRingCols = 32;

// Steps between a warp's bands: a row and one idle step, which clears the traces; so many that what the last warp's band
// leaves for the first warp's next one is SK + 1 steps old when it is read; and so many that the next band's column c
// is written to a ring's slot a group after the last column that shares the slot, at most (nx - 1) & ~31 further on, was
// read, SK + 1 steps after it was written.  (The last rule asks for idle steps where nx is 1 to 15 above a multiple of 32.)
__host__ __device__ constexpr int wave_period(int nx, int W, int SK) {
  const int a = nx + 1, b = W * (32 + SK), c = W > 1 ? ((nx - 1) & ~(kRingCols - 1)) + 2 * SK + 1 : 0;
  return a > b ? (a > c ? a : c) : (b > c ? b : c);
}

__device__ __forceinline__ void group_sync(int warps) {
  if (warps > 1) asm volatile("bar.sync 1, %0;" ::"r"(warps * 32) : "memory");
  else __syncwarp();
}

// BC: non-zero inflow on the x-faces (the right-hand side).  MINB: resident CTAs of 256 threads that the registers have
// to allow.  GT: the tables stay in global memory (problems with more regions than shared memory holds).
template <typename T, typename TI, typename ALG, int VW, int NV, int RPL, int PF, bool BC, int MINB, bool GT>
__global__ void __launch_bounds__(256, MINB) k_wave(SweepArgs a) {
  using V = Dv<T, VW>;
  constexpr int D = VW * NV, TW = ALG::TW, FW = ALG::FW, NC = ALG::NC, SK = PF;
  constexpr int HD = ALG::HD, RS = table_stride(HD + D * TW, sizeof(T));
  static_assert(!GT || VW == 1, "global tables are read one direction at a time");
  const SweepTask tk = a.tasks[blockIdx.x];
  if (a.active && !a.active[tk.b]) return;   // uniform for the CTA
  const InstInfo in = a.inst[tk.b];
  const int nx = in.nx, ny = in.ny, R = a.R, ndir = tk.n > 0 ? tk.n : D;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nb = (ny + 32 * RPL - 1) / (32 * RPL);
  const int W = min((int)(blockDim.x >> 5), nb);   // warps that have a band
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* tab = reinterpret_cast<T*>(smem_raw);          // [R + 1][RS]: [HD], cell tables [NV][TW][VW]; source factors [FW]
  T* cst = tab + (GT ? 0 : (size_t)(R + 1) * RS);   // [NV][NC][VW], padded to 4
  T* yfull = cst + ((NV * NC * VW + 3) & ~3);       // [nx][NV][2][VW] from the last warp's band to the first warp's next
  T* yring = yfull + (size_t)nx * D * 2;            // [W - 1][kRingCols][NV][2][VW] from a warp's band to the next warp's
  float4* sring = reinterpret_cast<float4*>(yring + (size_t)(W - 1) * kRingCols * D * 2);   // double-float: [W][PF][2][32]
  const UDir u0 = a.udir[tk.u0];
  const int sx = u0.sx, sy = u0.sy;
  // Stage the tables.  Directions beyond the task's own are zero (they carry no flux); so is the whole table R, which
  // lanes outside the mesh read: their traces become zero, the vacuum inflow of the row they enter next.
  const T* lin = reinterpret_cast<const T*>(a.linv) + ((size_t)tk.b * a.nu + tk.u0) * R * TW;
  const T* sgr = a.sig_s ? reinterpret_cast<const T*>(a.sig_s) + (size_t)tk.b * R : nullptr;
  if constexpr (!GT) {
    for (int e = threadIdx.x; e < (R + 1) * D * TW; e += blockDim.x) {
      const int k = e % TW, r = (e / TW) % (R + 1), d = e / (TW * (R + 1));
      tab[r * RS + HD + ((d / VW) * TW + k) * VW + d % VW] = r < R && d < ndir ? lin[((size_t)d * R + r) * TW + k] : (T)0;
    }
    if constexpr (FW > 0)
      for (int e = threadIdx.x; e < (R + 1) * FW; e += blockDim.x) {
        const int r = e / FW;
        const T f = r < R ? ALG::factor(e % FW, (double)sx, (double)sy) : (T)0;
        tab[r * RS + e % FW] = sgr && r < R ? f * sgr[r] : f;
      }
  }
  for (int d = threadIdx.x; d < D; d += blockDim.x) {
    T c[NC];
    if (d < ndir) {
      const UDir u = a.udir[tk.u0 + d];
      ALG::constants(u.ax / in.hx, u.ay / in.hy, u.w, c);
    } else {
      for (int k = 0; k < NC; ++k) c[k] = (T)0;
    }
    for (int k = 0; k < NC; ++k) cst[((d / VW) * NC + k) * VW + d % VW] = c[k];
  }
  // inflow traces of the constant g on the task's inflow faces (x face by the sign of Omega_x, y face by that of
  // Omega_y), zero on faces without inflow; the y-inflow of the first band goes where band 0 looks for it
  const double gtr = a.with_bc ? in.g * sqrt(in.hx * in.hy) : 0.0;
  T bx[2], by[2];
  ALG::boundary((a.inflow_mask & (sx > 0 ? 1 : 2)) ? gtr : 0.0, bx);
  ALG::boundary((a.inflow_mask & (sy > 0 ? 4 : 8)) ? gtr : 0.0, by);
  for (int e = threadIdx.x; e < nx * D * 2; e += blockDim.x) yfull[e] = by[(e / VW) & 1];
  if constexpr (std::is_same<T, dfloat>::value)   // lanes without a cell read their slots too
    for (int e = threadIdx.x; e < W * PF * 64; e += blockDim.x) sring[e] = make_float4(0.f, 0.f, 0.f, 0.f);
  __syncthreads();
  if (warp >= W) return;
  const TI* src = reinterpret_cast<const TI*>(a.src) + in.off;
  T* part = reinterpret_cast<T*>(a.partial) + (size_t)a.tasks_per_inst * in.off + (size_t)tk.t * in.ndof;
  constexpr int YC = D * 2;   // elements per column of a trace buffer
  const T* yin = warp == 0 ? yfull : yring + (size_t)(warp - 1) * kRingCols * YC;
  T* yout = warp == W - 1 ? yfull : yring + (size_t)warp * kRingCols * YC;
  const unsigned yin_s = (unsigned)__cvta_generic_to_shared(yin);
  const int min_ = warp == 0 ? -1 : kRingCols - 1, mout = warp == W - 1 ? -1 : kRingCols - 1;
  const int cx = nx / a.rx, cy = ny / a.ry, dx = sx > 0 ? 1 : -1;
  const int P = wave_period(nx, W, SK);
  const int last = (nb - 1) / W;
  // up to the last column of the mesh's last row: the last band of 40 rows has 8 lanes at work, not 32
  const int nsteps = last * P + (nb - 1 - last * W) * (32 + SK) + (ny - 1 - 32 * RPL * (nb - 1)) / RPL + nx;
  const unsigned mx = 0xffffffffu / (unsigned)cx + 1u, my = 0xffffffffu / (unsigned)cy + 1u;   // i / c = mulhi(i, m); c = 1: see div
  auto div = [](int i, unsigned m) { return m ? (int)__umulhi((unsigned)i, m) : i; };
  constexpr int RI = GT ? 1 : RS;   // table index per region
  const int rdx = sx > 0 ? RI : -RI, rowstep = 32 * RPL * W, dy = sy > 0 ? nx : -nx;
  auto cell0 = [&](int row) { return (sy > 0 ? row : ny - 1 - row) * nx + (sx > 0 ? 0 : nx - 1); };
  auto reg0 = [&](int row) {   // table of the row's first cell
    const int rr = div(row, my);
    return ((sy > 0 ? rr : a.ry - 1 - rr) * a.rx + (sx > 0 ? 0 : a.rx - 1)) * RI;
  };
  int row = 32 * RPL * warp + RPL * lane, col = -((32 + SK) * warp + lane);
  int cell = cell0(row), reg = reg0(row);
  int prow = row, pcol = col, pcell = cell;   // source prefetch, PF steps ahead
  // A double-float step is hundreds of instructions: unrolled, a group would not fit the instruction cache.  Its sources
  // then cannot rotate through registers (moving one waits for its load): they go to a ring in shared memory instead.
  constexpr bool kRing = std::is_same<T, dfloat>::value;
  auto fetch = [&](TI* dst, unsigned slot) {
#pragma unroll
    for (int r = 0; r < RPL; ++r)
      if ((unsigned)pcol < (unsigned)nx && prow + r < ny) {
        const TI* from = src + 4 * (long long)(pcell + dx * pcol + r * dy);
        if constexpr (kRing) {
          asm volatile("cp.async.cg.shared.global [%0], [%2], 16; cp.async.cg.shared.global [%1], [%3], 16;" ::"r"(slot),
                       "r"(slot + 512), "l"(from), "l"(from + 2)
                       : "memory");
        } else {
          Vec4<TI>::load(from, dst[4 * r], dst[4 * r + 1], dst[4 * r + 2], dst[4 * r + 3]);
        }
      }
    if constexpr (kRing) asm volatile("cp.async.commit_group;" ::: "memory");
    ++pcol;
    const bool wrap = pcol == P;
    pcol = wrap ? 0 : pcol;
    prow = wrap ? prow + rowstep : prow;
    pcell = wrap ? pcell + (sy > 0 ? rowstep * nx : -rowstep * nx) : pcell;
  };
  const unsigned ring = (unsigned)__cvta_generic_to_shared(sring) + (warp * PF * 64 + lane) * 16;   // this lane's slots
  TI q[kRing ? 1 : PF][4 * RPL];
  if constexpr (kRing) {
    static_assert(!kRing || (RPL == 1 && sizeof(TI) == 8), "a slot holds one cell");
#pragma unroll 1
    for (int k = 0; k < PF - 1; ++k) fetch(nullptr, ring + k * 1024);
  } else {
#pragma unroll
    for (int k = 0; k < PF; ++k) {
#pragma unroll
      for (int e = 0; e < 4 * RPL; ++e) q[k][e] = TI(0);
      fetch(q[k], 0);
    }
  }
  const unsigned neg[4] = {0u, sx > 0 ? 0u : 1u << 31, sy > 0 ? 0u : 1u << 31, sx * sy > 0 ? 0u : 1u << 31};
  // direction constants: in registers in FP32, re-read from shared memory where a value takes two registers
  constexpr bool kRegConst = sizeof(T) == 4;
  V creg[kRegConst ? NV : 1][NC];
  if constexpr (kRegConst)
#pragma unroll
    for (int v = 0; v < NV; ++v)
#pragma unroll
      for (int e = 0; e < NC; ++e) creg[v][e] = *reinterpret_cast<const V*>(cst + (v * NC + e) * VW);
  V X[RPL][NV][2], Y[NV][2];
#pragma unroll
  for (int v = 0; v < NV; ++v)
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      Y[v][e] = V::all((T)0);
#pragma unroll
      for (int r = 0; r < RPL; ++r) X[r][v][e] = V::all((T)0);
    }
  const bool first = lane == 0, tail = lane == 31;
  using BlkY = Blk<V, 2>;
  constexpr int UNR = kRing ? 1 : PF;
  for (int s0 = 0; s0 < nsteps; s0 += PF) {
#pragma unroll UNR
    for (int k0 = 0; k0 < PF; ++k0) {
      const int kk = kRing ? 0 : k0;
      const bool act = (unsigned)col < (unsigned)nx && row < ny;
      const int ro = act ? reg + rdx * div(col, mx) : (GT ? 0 : R * RS);
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        Y[v][0] = up1(Y[v][0]);
        Y[v][1] = up1(Y[v][1]);
      }
      {
        const unsigned take = first && act, at = yin_s + (unsigned)((col & min_) * YC * (int)sizeof(T));
#pragma unroll
        for (int v = 0; v < NV; ++v) load_traces(take, at + v * 2 * VW * (int)sizeof(T), Y[v]);
      }
      if constexpr (kRing) {   // the slot of the step before takes the source three steps ahead
        fetch(nullptr, ring + ((k0 + PF - 1) % PF) * 1024);
        asm volatile("cp.async.wait_group %0;" ::"n"(PF - 1) : "memory");
      }
      {
        if constexpr (BC) {
#pragma unroll
          for (int v = 0; v < NV; ++v)
#pragma unroll
            for (int e = 0; e < 2; ++e)
#pragma unroll
              for (int r = 0; r < RPL; ++r)
                if (col == 0) X[r][v][e] = V::all(bx[e]);
        }
        constexpr int FB = FW > 0 ? FW : 1;
        Blk<T, FB> sg;
        if constexpr (FW > 0) {
          if constexpr (GT) sg.v[0] = sgr ? sgr[ro] : (T)1;
          else sg = *reinterpret_cast<const Blk<T, FB>*>(tab + ro);
        }
        V S[RPL][4], acc[RPL][4];
#pragma unroll
        for (int r = 0; r < RPL; ++r) {
          T t[4], Sr[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) t[e] = (T)q[kk][4 * r + e];
          if constexpr (kRing) {
            const float4* sl = sring + (warp * PF + k0) * 64 + lane;
            const float4 v0 = sl[0], v1 = sl[32];
            t[0] = dfloat(v0.x, v0.y);
            t[1] = dfloat(v0.z, v0.w);
            t[2] = dfloat(v1.x, v1.y);
            t[3] = dfloat(v1.z, v1.w);
          }
          ALG::source(t, sg.v, neg, Sr);
#pragma unroll
          for (int e = 0; e < 4; ++e) S[r][e] = V::all(Sr[e]);
        }
        if constexpr (!kRing) fetch(q[kk], 0);
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          using BlkM = Blk<V, TW>;
          BlkM m;
          if constexpr (GT) m = *reinterpret_cast<const BlkM*>(lin + ((size_t)min(v, ndir - 1) * R + ro) * TW);
          else m = *reinterpret_cast<const BlkM*>(tab + ro + HD + v * TW * VW);
          V c[NC];
#pragma unroll
          for (int e = 0; e < NC; ++e) {
            if constexpr (kRegConst) c[e] = creg[v][e];
            else c[e] = *reinterpret_cast<const V*>(cst + (v * NC + e) * VW);
          }
#pragma unroll
          for (int r = 0; r < RPL; ++r) ALG::cell(S[r], X[r][v], Y[v], m.v, c, acc[r], v == 0);
        }
#pragma unroll
        for (int r = 0; r < RPL; ++r) {
          T c4[4], o[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) c4[e] = acc[r][e].sum();
          ALG::from_basis(c4, o);
          if constexpr (sizeof(T) == 4) {   // a select with a negated operand; in FP64 the negation would be an instruction
            o[1] = sx > 0 ? o[1] : -o[1];
            o[2] = sy > 0 ? o[2] : -o[2];
            o[3] = sx * sy > 0 ? o[3] : -o[3];
          } else {
#pragma unroll
            for (int e = 1; e < 4; ++e) o[e] = flip(o[e], neg[e]);
          }
          if (act && (RPL == 1 || row + r < ny))
            Vec4<T>::store(part + 4 * (long long)(cell + dx * col + r * dy), o[0], o[1], o[2], o[3]);
        }
        if (tail && act) {
#pragma unroll
          for (int v = 0; v < NV; ++v) {
            BlkY y;
            y.v[0] = Y[v][0];
            y.v[1] = Y[v][1];
            *reinterpret_cast<BlkY*>(yout + (col & mout) * YC + v * 2 * VW) = y;
          }
        }
      }
      // lanes without a cell hand on the vacuum inflow of the row they enter next (else the zero table sees to that)
      if (GT && !act) {
#pragma unroll
        for (int v = 0; v < NV; ++v)
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            Y[v][e] = V::all((T)0);
#pragma unroll
            for (int r = 0; r < RPL; ++r) X[r][v][e] = V::all((T)0);
          }
      }
      ++col;
      const bool wrap = col == P;
      col = wrap ? 0 : col;
      row = wrap ? row + rowstep : row;
      cell = wrap ? cell + (sy > 0 ? rowstep * nx : -rowstep * nx) : cell;
      reg = wrap ? reg0(row) : reg;
    }
    group_sync(W);
  }
  if constexpr (kRing) asm volatile("cp.async.wait_all;" ::: "memory");
}

// ------------------------------------------------------------------------------------------------- launch
static void mesh_max(const rte_problem* p, int* nx, int* ny) {
  *nx = *ny = 0;
  for (int b = 0; b < p->B; ++b) {
    *nx = std::max(*nx, p->nx[b]);
    *ny = std::max(*ny, p->ny[b]);
  }
}

constexpr size_t kMaxSmem = 227 * 1024;

// Shared memory of a CTA.  tables: with the region tables, else with these left in global memory.
static size_t shape_smem(const rte_problem* p, int prec, WaveShape s, bool tables) {
  using F = Rot<float>;
  using W = Legendre<double, true>;
  int nx, ny;
  mesh_max(p, &nx, &ny);
  const bool f32 = prec == PREC_F32;
  const int nc = f32 ? F::NC : (prec == PREC_F64 ? W::NC : Scaled::NC);
  const int rs = f32 ? table_stride(F::HD + s.D * F::TW, 4)
                     : (prec == PREC_F64 ? table_stride(W::HD + s.D * (s.D > 2 ? Nine<double, true>::TW : W::TW), 8)
                                         : table_stride(s.D * Scaled::TW, 8));
  const size_t elems = (tables ? (size_t)(p->R + 1) * rs : 0) + ((s.D * nc + 3) & ~3) +
                       ((size_t)nx + (s.W - 1) * kRingCols) * s.D * 2;
  return elems * (f32 ? 4 : 8) + (prec == PREC_DF ? (size_t)s.W * 4 * 1024 : 0);   // and the ring of sources
}

// FP64 and double-float tables (144 and 80 bytes a region with one direction) stay in global memory where shared memory
// does not hold them: 1,600 and 2,800 regions and more with one direction, 690 and 670 with four.
static bool global_tables(const rte_problem* p, int prec, WaveShape s) {
  return prec != PREC_F32 && shape_smem(p, prec, s, true) > kMaxSmem;
}

size_t wave_smem(const rte_problem* p, int prec, WaveShape s) {
  return shape_smem(p, prec, s, !global_tables(p, prec, s));
}

template <typename T_, typename TI, typename ALG, int VW, int NV, int RPL, int PF, bool BC, int MINB, bool GT>
struct WaveKernel {
  static constexpr auto fn = k_wave<T_, TI, ALG, VW, NV, RPL, PF, BC, MINB, GT>;
  static int launch(const SweepArgs& a, int W, size_t smem, cudaStream_t st) {
    static std::atomic<size_t> granted[kMaxDevices];
    RTE_TRY(grant_smem(fn, smem, granted));
    fn<<<a.ntasks, W * 32, smem, st>>>(a);
    count_launch();
    RTE_CHECK_CUDA(cudaGetLastError());
    return RTE_OK;
  }
  static int regs() {   // a thread's registers, a property of the compiled kernel
    static std::atomic<int> n{0};
    if (n.load() == 0) {
      cudaFuncAttributes at;
      if (cudaFuncGetAttributes(&at, fn) != cudaSuccess) {
        cudaGetLastError();
        return 128;
      }
      n.store((at.numRegs + 7) & ~7);
    }
    return n.load();
  }
};

// The kernel of a shape: f(WaveKernel<...>{}), or `none` where it is not built.  FP32 sweeps of FP64 vectors are the
// right-hand side and the inner solves with FP64 Krylov vectors.  sig: an FP64 source that is still to be multiplied by
// Sigma_s.
template <bool BC, typename F>
static int with_kernel(int prec, WaveShape s, bool in64, bool sig, bool gt, int none, F&& f) {
  const int shape = s.D * 10 + s.rpl;
  if (prec == PREC_F32) {
    using A = Rot<float>;
    if (BC || in64) {
      switch (shape) {
        case 11: return f(WaveKernel<float, double, A, 1, 1, 1, 8, true, 2, false>{});
        case 21: return f(WaveKernel<float, double, A, 2, 1, 1, 8, true, 2, false>{});
        case 41: return f(WaveKernel<float, double, A, 2, 2, 1, 8, true, 2, false>{});
        case 81: return f(WaveKernel<float, double, A, 2, 4, 1, 4, true, 2, false>{});
        case 121: return f(WaveKernel<float, double, A, 2, 6, 1, 4, true, 1, false>{});
        case 161: return f(WaveKernel<float, double, A, 2, 8, 1, 4, true, 1, false>{});
        case 82: return f(WaveKernel<float, double, A, 2, 4, 2, 4, true, 1, false>{});
      }
    } else {
      switch (shape) {
        case 11: return f(WaveKernel<float, float, A, 1, 1, 1, 8, false, 2, false>{});
        case 21: return f(WaveKernel<float, float, A, 2, 1, 1, 8, false, 2, false>{});
        case 41: return f(WaveKernel<float, float, A, 2, 2, 1, 8, false, 2, false>{});
        case 81: return f(WaveKernel<float, float, A, 2, 4, 1, 4, false, 2, false>{});
        case 121: return f(WaveKernel<float, float, A, 2, 6, 1, 4, false, 1, false>{});
        case 161: return f(WaveKernel<float, float, A, 2, 8, 1, 4, false, 1, false>{});
        case 82: return f(WaveKernel<float, float, A, 2, 4, 2, 4, false, 1, false>{});
      }
    }
  } else if (prec == PREC_F64) {
    auto pick = [&](auto few, auto many) {   // one and two directions a task, three and more
      using A = decltype(few);
      using M = decltype(many);
      switch (shape * 2 + gt) {
        case 22: return f(WaveKernel<double, double, A, 1, 1, 1, 4, BC, 2, false>{});
        case 42: return f(WaveKernel<double, double, A, 1, 2, 1, 4, BC, 2, false>{});
        case 62: return f(WaveKernel<double, double, M, 1, 3, 1, 4, BC, 2, false>{});
        case 82: return f(WaveKernel<double, double, M, 1, 4, 1, 4, BC, 1, false>{});
        case 23: return f(WaveKernel<double, double, A, 1, 1, 1, 4, BC, 1, true>{});
        case 43: return f(WaveKernel<double, double, A, 1, 2, 1, 4, BC, 1, true>{});
        case 83: return f(WaveKernel<double, double, M, 1, 4, 1, 4, BC, 1, true>{});
      }
      return none;
    };
    if constexpr (!BC)
      if (sig) return pick(Legendre<double, true>{}, Nine<double, true>{});
    return pick(Legendre<double, false>{}, Nine<double, false>{});
  } else if (!BC) {
    using A = Scaled;
    switch (shape * 2 + gt) {
      case 22: return f(WaveKernel<dfloat, dfloat, A, 1, 1, 1, 4, false, 2, false>{});
      case 42: return f(WaveKernel<dfloat, dfloat, A, 1, 2, 1, 4, false, 2, false>{});
      case 82: return f(WaveKernel<dfloat, dfloat, A, 1, 4, 1, 4, false, 1, false>{});
      case 23: return f(WaveKernel<dfloat, dfloat, A, 1, 1, 1, 4, false, 1, true>{});
    }
  }
  return none;
}

// Registers a thread of a shape takes (0: not built): they set how many warps an SM holds.
static int shape_regs(const rte_problem* p, int prec, WaveShape s) {
  return with_kernel<false>(prec, s, false, false, global_tables(p, prec, s), 0, [](auto k) { return decltype(k)::regs(); });
}

static bool shape_built(const rte_problem* p, int prec, WaveShape s) {
  return with_kernel<false>(prec, s, false, false, global_tables(p, prec, s), 0, [](auto) { return 1; }) != 0;
}

bool wave_shape_ok(const rte_problem* p, int prec, WaveShape s) {
  if (s.W < 1 || s.W > 8 || !shape_built(p, prec, s) || wave_smem(p, prec, s) > kMaxSmem) return false;
  if (s.rpl == 2)   // the two rows of a lane share a table: they have to lie in one region in both sweep directions
    for (int b = 0; b < p->B; ++b)
      if (p->ny[b] % 2 || (p->ny[b] / p->ry) % 2) return false;
  return true;
}

// Estimated time of an operator sweep with a shape, in SM cycles; only ratios matter.  SM 0 gets tasks 0, SMs, 2 SMs, ...
// of the list (longest first), as many at a time as its registers and shared memory hold; its resident warps advance in
// step, one step taking the pipe cycles of all of them or the latency of one alone, whichever is longer.  Per warp and
// step, measured: FP32 10 D + 40 cycles of the load/store data pipe (tables, shuffles; 13 D + 30 with two rows a lane),
// the pipe that fills up first, of which single-warp tasks reach 0.65 and wider ones 0.75, 50 D + 300 alone (1750 with
// two rows); FP64 19 cycles of the SM's FP64 unit for each of 32 D instructions, 70 alone; double-float 356 D + 160
// instructions, 0.85 a cycle and SM quarter, 0.5 alone.  The partial fluxes, written and read once, are added at the copy
// bandwidth.
static double wave_cost(const rte_problem* p, int prec, WaveShape s, int sms, const std::vector<int>& order) {
  const int SK = 4, per_sm = 65536 / (shape_regs(p, prec, s) * 32);
  const size_t smem = wave_smem(p, prec, s) + 1024;
  const size_t slots = std::max(1, std::min(per_sm / s.W, (int)(kMaxSmem / smem)));
  int chunks = 0;
  for (int q = 0; q < 4; ++q) chunks += (p->quad_start[q + 1] - p->quad_start[q] + s.D - 1) / s.D;
  double pipe, alone;
  if (prec == PREC_F32) {
    pipe = (s.rpl == 2 ? 13.0 * s.D + 30.0 : 10.0 * s.D + 40.0) / (s.W == 1 ? 0.65 : 0.75);
    alone = s.rpl == 2 ? 1750.0 : 50.0 * s.D + 300.0;
  } else if (prec == PREC_F64) {
    const double instr = 32.0 * s.D;
    pipe = 19.0 * instr;
    alone = 70.0 * instr;
  } else {
    pipe = (356.0 * s.D + 160.0) / 3.4;   // of warps in multiples of four
    alone = (356.0 * s.D + 160.0) / 0.5;
  }
  struct Run {
    double steps;
    int W;
  };
  std::vector<Run> queue, held;
  for (long long i = 0; i < (long long)p->B * chunks; i += sms) {
    const int b = order[i / chunks];
    const int nb = (p->ny[b] + 32 * s.rpl - 1) / (32 * s.rpl), W = std::min(s.W, nb), last = (nb - 1) / W;
    queue.push_back({(double)last * wave_period(p->nx[b], W, SK) + (nb - 1 - last * W) * (32 + SK) +
                         (p->ny[b] - 1 - 32 * s.rpl * (nb - 1)) / s.rpl + p->nx[b], W});
  }
  double t = 0.0;
  for (size_t next = 0; next < queue.size() || !held.empty();) {
    while (held.size() < slots && next < queue.size()) held.push_back(queue[next++]);
    double least = held[0].steps;
    int warps = 0;
    for (const Run& r : held) {
      least = std::min(least, r.steps);
      warps += r.W;
    }
    if (prec == PREC_DF) warps = (warps + 3) & ~3;
    t += least * std::max(alone, warps * pipe);
    for (Run& r : held) r.steps -= least;
    held.erase(std::remove_if(held.begin(), held.end(), [](const Run& r) { return r.steps <= 0.5; }), held.end());
  }
  return t + 2.0 * (double)chunks * (double)p->ntot * (prec == PREC_F32 ? 4 : 8) / 3300.0;   // bytes a cycle at 6.7 TB/s
}

// the instances in the order of the task list: most cells first
static std::vector<int> task_order(const rte_problem* p) {
  std::vector<int> order(p->B);
  for (int b = 0; b < p->B; ++b) order[b] = b;
  std::stable_sort(order.begin(), order.end(),
                   [&](int x, int y) { return (long long)p->nx[x] * p->ny[x] > (long long)p->nx[y] * p->ny[y]; });
  return order;
}

static int device_sms() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    cudaGetLastError();
  return std::max(1, sms);
}

std::vector<WaveShape> wave_shapes(const rte_problem* p, int prec, int keep) {
  const int sms = device_sms();
  const std::vector<int> order = task_order(p);
  int maxny = 0, maxq = 0;
  for (int b = 0; b < p->B; ++b) maxny = std::max(maxny, p->ny[b]);
  for (int q = 0; q < 4; ++q) maxq = std::max(maxq, p->quad_start[q + 1] - p->quad_start[q]);
  std::vector<std::pair<double, WaveShape>> all;
  for (int D : {1, 2, 3, 4, 8, 12, 16})
    for (int W : {1, 2, 4, 8})
      for (int rpl : {1, 2}) {
        const WaveShape s{D, W, rpl};
        if (W > 1 && W / 2 >= (maxny + 32 * rpl - 1) / (32 * rpl)) continue;   // half of the warps without a band
        if (D > 1 && D >= 2 * maxq) continue;
        if (wave_shape_ok(p, prec, s)) all.push_back({wave_cost(p, prec, s, sms, order), s});
      }
  std::stable_sort(all.begin(), all.end(), [](const auto& x, const auto& y) { return x.first < y.first; });
  std::vector<WaveShape> out;
  for (size_t i = 0; i < all.size() && (int)i < keep; ++i) out.push_back(all[i].second);
  return out;
}

WaveShape wave_shape_for(const rte_problem* p, int prec, int D) {
  WaveShape best{D, 1, 1};
  double cost = 1e300;
  const int sms = device_sms();
  const std::vector<int> order = task_order(p);
  for (int W : {1, 2, 4, 8}) {
    const WaveShape s{D, W, 1};
    if (!wave_shape_ok(p, prec, s)) continue;
    const double c = wave_cost(p, prec, s, sms, order);
    if (c < cost) {
      cost = c;
      best = s;
    }
  }
  return best;
}

int launch_wave(const rte_problem* p, int prec, WaveShape s, bool in64, const SweepArgs& args, cudaStream_t st) {
  if (!wave_shape_ok(p, prec, s)) {
    set_error("sweep: shared-memory table too large for this mesh/region count");
    return RTE_ERR_UNSUPPORTED;
  }
  SweepArgs a = args;
  if (prec == PREC_F32) a.linv = p->d_rot32.p;   // else the cell inverses of the arithmetic
  if (prec == PREC_F64 && s.D > 2) a.linv = p->d_inv64.p;
  const size_t smem = wave_smem(p, prec, s);
  auto run = [&](auto k) { return decltype(k)::launch(a, s.W, smem, st); };
  const bool gt = global_tables(p, prec, s);
  return a.with_bc ? with_kernel<true>(prec, s, in64, false, gt, RTE_ERR_UNSUPPORTED, run)
                   : with_kernel<false>(prec, s, in64, a.sig_s != nullptr, gt, RTE_ERR_UNSUPPORTED, run);
}

}  // namespace rte

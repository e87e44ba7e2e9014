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
// 1, N_x, N_y, N_x N_y, and two bases make that cheap:
//  * Rot (FP32): both axes turned by 45 degrees, x' = (x_0 + x_1, x_1 - x_0) / sqrt2, an orthogonal change of basis.
//    There N = [[0, a], [-1/a, 0]], a^2 = 2 + sqrt3, the outflow functional is (a, 1/a) and the inflow vector
//    -(1/a, a).  With the second component of each axis scaled by q = 1/a^2, traces in units of a, the inflow enters
//    both components of a pair with the same weight -alpha (or -beta), the outflow is a plain sum, and L^{-1} has
//    eight distinct entries: 8 + 16 + 4 multiply-adds and adds and 4 for the quadrature, against 9 + 16 + 4 + 4 and
//    sixteen entries in the Legendre basis, with the same rounding errors.
//  * Modal (FP64, double-float): the eigenbasis of N on both axes.  A real 4-vector becomes two complex numbers
//    A (modes (i, i)) and B (modes (i, -i)) on which L is multiplication by a complex number:
//    A = G_A (S_A + alpha X + beta Y), B = G_B (S_B + alpha conj X + beta rho Y), X' = A + conj B, Y' = A + B:
//    24 multiply-adds and adds and four table entries.  The eigenbasis is not orthogonal (condition number 3.7): with
//    tables rounded once the FP64 apply is as close to 64-bit reference values as in the Legendre basis (7.5e-16 against
//    4.9e-16 to 8.1e-16), but in FP32 the error would grow 1.7x, so FP32 keeps Rot (2.1e-7 either way).
// The source is brought to the basis, and the summed flux back, once per cell and task (about 30 operations over D
// directions).
//
// FP32 runs pairs of directions in the packed multiply-add (fma.rn.f32x2): half the issue slots at the same rate.
//
// Bounds and measurements (one operator apply with the sum of its partial fluxes, GB300; before: Legendre basis, sixteen
// table entries per direction and region, D <= 8, one warp per task or per band).  FP32, 64 x 256^2, 192 directions,
// 8 x 8 regions: 2.08 -> 0.98 ms (D = 12, W = 2; 63 % of the load/store data pipe, 47 % of the FMA pipe); 256 instances
// on 32^2, 64^2 and 128^2, 128 directions: 0.672 -> 0.331 ms (D = 8, two rows a lane: each table and shuffle serves two
// cells); one 64^2 instance: 36.8 -> 28.8 us (latency of 131 steps).  FP64 is bound by the FP64 unit (19 SM cycles a warp
// instruction), so by instructions per cell and direction: 7.93 -> 6.73 ms on the 256 instances, 0.919 -> 0.726 ms on
// 10 x 80^2 with CL(30, 6), where D = 3 now divides quadrants of 24 and 21 directions (before: D = 1).  Double-float is
// bound by FP32 issue: 3.61 -> 2.00 ms on 16 x 256^2 (sums of products with one renormalisation each, and the step loop
// not unrolled: unrolled it missed the instruction cache, 3.48 ms).
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

// ------------------------------------------------------------------------------------------- cell algebras
// Sums of products.  FP64: multiply-adds.  Double-float: the high parts go through two-sums, what these miss and the
// low parts are added up on the side, and one renormalisation ends the sum (the compensated dot product of Ogita, Rump
// and Oishi, SIAM J. Sci. Comput. 26, 2005): 12 operations a term against 18 for a product and a sum of pairs.
template <typename T>
struct Sum {
  T v;
  __device__ __forceinline__ explicit Sum(T a) : v(a) {}
  __device__ __forceinline__ Sum(T a, T b) : v(a * b) {}
  __device__ __forceinline__ Sum add(T a, T b) const { return Sum(v + a * b); }
  __device__ __forceinline__ Sum sub(T a, T b) const { return Sum(v - a * b); }
  __device__ __forceinline__ T get() const { return v; }
};
template <>
struct Sum<dfloat> {
  float s, e;
  __device__ __forceinline__ explicit Sum(dfloat a) : s(a.hi), e(a.lo) {}
  __device__ __forceinline__ Sum(dfloat a, dfloat b) {
    s = __fmul_rn(a.hi, b.hi);
    e = __fmaf_rn(a.lo, b.hi, __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.hi, b.hi, -s)));
  }
  __device__ __forceinline__ Sum add(dfloat a, dfloat b) const {
    Sum r(a, b);
    const float t = __fadd_rn(s, r.s), bb = __fsub_rn(t, s);
    const float er = __fadd_rn(__fsub_rn(s, __fsub_rn(t, bb)), __fsub_rn(r.s, bb));
    r.s = t;
    r.e = __fadd_rn(e, __fadd_rn(er, r.e));
    return r;
  }
  __device__ __forceinline__ Sum sub(dfloat a, dfloat b) const { return add(dfloat(-a.hi, -a.lo), b); }
  __device__ __forceinline__ dfloat get() const { return df_renorm(s, e); }
};

template <typename T>
struct Rot {
  static constexpr int TW = 8;   // table entries per direction and region
  static constexpr int NC = 3;   // constants per direction: -alpha, -beta, omega
  static constexpr double A2 = 3.7320508075688772935, Q = 0.26794919243112270647;
  // factors of the source's four Legendre components before to_basis, for reflection signs fx, fy
  __device__ static T factor(int k, double fx, double fy) {
    return (T)(0.5 * ((k & 1) ? fx : 1.0) * ((k & 2) ? fy : 1.0));
  }
  __device__ __forceinline__ static void to_basis(const T* t, T* S) {
    const T u = t[0] + t[3], d = t[3] - t[0], e = t[1] + t[2], f = t[1] - t[2];
    S[0] = u + e;
    S[1] = (T)Q * (d + f);
    S[2] = (T)Q * (d - f);
    S[3] = (T)(Q * Q) * (u - e);
  }
  __device__ __forceinline__ static void from_basis(const T* c, T* s) {
    const T e0 = (T)0.5 * c[0], e1 = (T)(0.5 * A2) * c[1], e2 = (T)(0.5 * A2) * c[2], e3 = (T)(0.5 * A2 * A2) * c[3];
    const T u = e0 + e3, v = e1 + e2, w = e0 - e3, z = e1 - e2;
    s[0] = u - v;
    s[1] = w + z;
    s[2] = w - z;
    s[3] = u + v;
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

// Constants of the eigenbasis: u = (1, mu), mu = -(1 + i sqrt2) / sqrt3, the left eigenvector of K to 2 + i sqrt2; both
// axes scaled by c / 2 = (1 + 2 i sqrt2) / 2, which makes both outflow functionals (1, 1); sources divided by
// kappa = c (2 + i sqrt2) / 2 = -1 + 5 i / sqrt2, which makes the x-inflow weights alpha; rho = conj(kappa) / kappa.
template <typename T>
struct Modal {
  static constexpr int TW = 4;
  static constexpr int NC = 5;   // alpha, beta, beta Re rho, beta Im rho, omega
  __device__ static T factor(int k, double fx, double fy) {
    return (T)(((k & 1) ? fx : 1.0) * ((k & 2) ? fy : 1.0));
  }
  __device__ __forceinline__ static void to_basis(const T* t, T* S) {
    const T e = t[0] + t[3];
    S[0] = (T)0.5 * (t[0] - t[3]);
    S[1] = Sum<T>((T)0.35355339059327376220, e).add((T)(-0.61237243569579452455), t[1] + t[2]).get();
    S[2] = Sum<T>((T)(-1.0 / 6.0), e).add((T)(-0.38490017945975050967), t[1]).add((T)0.57735026918962576451, t[2]).get();
    S[3] = Sum<T>((T)(-0.58925565098878960367), e).add((T)0.47628967220784018576, t[1])
               .add((T)0.20412414523193150818, t[2]).get();
  }
  // (Re A, R, Im X', Im Y') -> Legendre components, from A = (c/2)^2 (u (x) u) p, B = |c/2|^2 (u (x) conj u) p
  __device__ __forceinline__ static void from_basis(const T* c, T* s) {
    const T z = c[2] + c[3], d = c[3] - c[2];
    s[0] = Sum<T>((T)(-2.0 / 9.0), c[0]).add((T)(1.0 / 3.0), c[1]).add((T)0.15713484026367723, z).get();
    s[3] = Sum<T>((T)(-2.0 / 27.0), c[0]).add((T)(1.0 / 3.0), c[1]).add((T)(-0.10475656017578482), z).get();
    const T f = Sum<T>((T)0.12830005981991683, c[0]).add((T)0.19245008972987526, c[1]).add((T)0.04536092116265145, z).get();
    const T h = (T)0.13608276348795434 * d;
    s[1] = f - h;
    s[2] = f + h;
  }
  __device__ static void boundary(double g, T* t) {
    t[0] = (T)(0.5 * g);
    t[1] = (T)(1.4142135623730950488 * g);
  }
  __device__ static void constants(double al, double be, double w, T* c) {
    c[0] = (T)al;
    c[1] = (T)be;
    c[2] = (T)(-23.0 * be / 27.0);
    c[3] = (T)(0.52378280087892411 * be);
    c[4] = (T)w;
  }
  template <typename V>
  __device__ __forceinline__ static void cell(const V* S, V* X, V* Y, const V* m, const V* c, V* acc, bool zero) {
    const T a = c[0].x, b = c[1].x, b1 = c[2].x, b2 = c[3].x, w = c[4].x;
    const T x0 = X[0].x, x1 = X[1].x, y0 = Y[0].x, y1 = Y[1].x;
    const T ar = Sum<T>(S[0].x).add(a, x0).add(b, y0).get(), ai = Sum<T>(S[1].x).add(a, x1).add(b, y1).get();
    const T br = Sum<T>(S[2].x).add(a, x0).add(b1, y0).sub(b2, y1).get();
    const T bi = Sum<T>(S[3].x).sub(a, x1).add(b1, y1).add(b2, y0).get();
    const T Ar = Sum<T>(m[0].x, ar).sub(m[1].x, ai).get(), Ai = Sum<T>(m[0].x, ai).add(m[1].x, ar).get();
    const T R = Sum<T>(Ar).add(m[2].x, br).sub(m[3].x, bi).get(), Bi = Sum<T>(m[2].x, bi).add(m[3].x, br).get();
    X[0].x = Y[0].x = R;
    X[1].x = Ai - Bi;
    Y[1].x = Ai + Bi;
    acc[0].x = zero ? w * Ar : Sum<T>(acc[0].x).add(w, Ar).get();
    acc[1].x = zero ? w * R : Sum<T>(acc[1].x).add(w, R).get();
    acc[2].x = zero ? w * X[1].x : Sum<T>(acc[2].x).add(w, X[1].x).get();
    acc[3].x = zero ? w * Y[1].x : Sum<T>(acc[3].x).add(w, Y[1].x).get();
  }
};

// The Legendre basis itself: no transforms, sixteen table entries (the cell inverses), 32 D + 4 operations a cell against
// 24 D + 30.  FP64 tasks of one or two directions, which do not pay for the eigenbasis's transforms (26 x (64 x 22), 28
// directions in quadrants of 8 and 6, D = 1: 271 us in the eigenbasis, 190 us here).
template <typename T>
struct Legendre {
  static constexpr int TW = 16;
  static constexpr int NC = 5;   // alpha, beta, sqrt3 alpha, sqrt3 beta, omega
  __device__ static T factor(int k, double fx, double fy) {
    return (T)(((k & 1) ? fx : 1.0) * ((k & 2) ? fy : 1.0));
  }
  __device__ __forceinline__ static void to_basis(const T* t, T* S) {
#pragma unroll
    for (int e = 0; e < 4; ++e) S[e] = t[e];
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

// Unevaluated sums of two doubles, for the tables alone (two-sum and two-product as in dfloat.cuh)
struct Dd {
  double h, l;
};
__device__ Dd dd_sum(double a, double b) {
  const double s = __dadd_rn(a, b), t = __dsub_rn(s, a);
  return Dd{s, __dadd_rn(__dsub_rn(a, __dsub_rn(s, t)), __dsub_rn(b, t))};
}
__device__ Dd dd_add(Dd a, Dd b) {
  const Dd s = dd_sum(a.h, b.h);
  return dd_sum(s.h, __dadd_rn(s.l, __dadd_rn(a.l, b.l)));
}
__device__ Dd dd_mul(Dd a, Dd b) {
  const double p = __dmul_rn(a.h, b.h);
  return dd_sum(p, __fma_rn(a.l, b.h, __fma_rn(a.h, b.l, __fma_rn(a.h, b.h, -p))));
}
__device__ double dd_div(Dd a, Dd b) {   // a / b to double
  const double q = __ddiv_rn(a.h, b.h);
  const Dd p = dd_mul(Dd{q, 0.0}, b), r = dd_add(a, Dd{-p.h, -p.l});
  return __dadd_rn(q, __ddiv_rn(r.h, b.h));
}

// Tables per (instance, unique direction, region): Rot FP32 [8], Modal FP64 [4] and double-float [4] pairs.
// l_1 = c_0 + i sqrt2 (alpha + beta), l_2 = c_0 + i sqrt2 (alpha - beta), c_0 = 2 (alpha + beta) + sigma_t, are the
// eigenvalues of L on (i, i) and (i, -i); L^{-1} = g + g_x N_x + g_y N_y + g_xy N_x N_y follows from 1 / l_1, 1 / l_2.
__global__ void k_wave_tables(int B, int nu, int R, const InstInfo* inst, const UDir* ud, const double* sig_t,
                              float* rot, double* modal, float* modal_df) {
  const long long tid = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (tid >= (long long)B * nu * R) return;
  const int r = (int)(tid % R), u = (int)((tid / R) % nu), b = (int)(tid / ((long long)R * nu));
  const double al = ud[u].ax / inst[b].hx, be = ud[u].ay / inst[b].hy, sg = sig_t[(size_t)b * R + r];
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
  // G = kappa / l, rounded once: what the rounding of the tables loses adds up along a ray
  const Dd s2d{1.4142135623730951, -9.667293313452913e-17}, kid{3.5355339059327378, -1.3066003037380717e-16};
  const Dd sum = dd_sum(al, be), dif = dd_sum(al, -be);
  const Dd c0d = dd_add(Dd{2.0 * sum.h, 2.0 * sum.l}, Dd{sg, 0.0});
  const Dd i1d = dd_mul(s2d, sum), i2d = dd_mul(s2d, dif);
  const Dd n1d = dd_add(dd_mul(c0d, c0d), dd_mul(i1d, i1d)), n2d = dd_add(dd_mul(c0d, c0d), dd_mul(i2d, i2d));
  const Dd nc{-c0d.h, -c0d.l};
  const double m[4] = {dd_div(dd_add(dd_mul(kid, i1d), nc), n1d), dd_div(dd_add(dd_mul(kid, c0d), i1d), n1d),
                       dd_div(dd_add(dd_mul(kid, i2d), nc), n2d), dd_div(dd_add(dd_mul(kid, c0d), i2d), n2d)};
  for (int k = 0; k < 4; ++k) {
    modal[tid * 4 + k] = m[k];
    const float h = (float)m[k];
    modal_df[2 * (tid * 4 + k)] = h;
    modal_df[2 * (tid * 4 + k) + 1] = (float)(m[k] - (double)h);
  }
}

int build_wave_tables(rte_problem* p) {
  const long long n = (long long)p->B * p->nu * p->R;
  k_wave_tables<<<(unsigned)((n + 127) / 128), 128>>>(p->B, p->nu, p->R, p->d_inst.p, p->d_udir.p, p->d_sig_t.p,
                                                      p->d_rot32.p, p->d_modal64.p, p->d_modal_df.p);
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
constexpr int kRing = 32;

// Steps between a warp's bands: a row and one idle step, which clears the traces; so many that what the last warp's band
// leaves for the first warp's next one is SK + 1 steps old when it is read; and so many that the next band's column c
// is written to a ring's slot a group after the last column that shares the slot, at most (nx - 1) & ~31 further on, was
// read, SK + 1 steps after it was written.  (The last rule asks for idle steps where nx is 1 to 15 above a multiple of 32.)
__host__ __device__ constexpr int wave_period(int nx, int W, int SK) {
  const int a = nx + 1, b = W * (32 + SK), c = W > 1 ? ((nx - 1) & ~(kRing - 1)) + 2 * SK + 1 : 0;
  return a > b ? (a > c ? a : c) : (b > c ? b : c);
}

__device__ __forceinline__ void group_sync(int warps) {
  if (warps > 1) asm volatile("bar.sync 1, %0;" ::"r"(warps * 32) : "memory");
  else __syncwarp();
}

// BC: non-zero inflow on the x-faces (the right-hand side).  MINB: resident CTAs of 256 threads that the registers have
// to allow.
template <typename T, typename TI, typename ALG, int VW, int NV, int RPL, int PF, bool BC, int MINB>
__global__ void __launch_bounds__(256, MINB) k_wave(SweepArgs a) {
  using V = Dv<T, VW>;
  constexpr int D = VW * NV, TW = ALG::TW, NC = ALG::NC, SK = PF;
  constexpr int RS = table_stride(4 + D * TW, sizeof(T));
  const SweepTask tk = a.tasks[blockIdx.x];
  if (a.active && !a.active[tk.b]) return;   // uniform for the CTA
  const InstInfo in = a.inst[tk.b];
  const int nx = in.nx, ny = in.ny, R = a.R, ndir = tk.n > 0 ? tk.n : D;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nb = (ny + 32 * RPL - 1) / (32 * RPL);
  const int W = min((int)(blockDim.x >> 5), nb);   // warps that have a band
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* tab = reinterpret_cast<T*>(smem_raw);          // [R + 1][RS]: source factors [4], cell tables [NV][TW][VW]
  T* cst = tab + (size_t)(R + 1) * RS;              // [NV][NC][VW], padded to 4
  T* yfull = cst + ((NV * NC * VW + 3) & ~3);       // [nx][NV][2][VW] from the last warp's band to the first warp's next
  T* yring = yfull + (size_t)nx * D * 2;            // [W - 1][kRing][NV][2][VW] from a warp's band to the next warp's
  const UDir u0 = a.udir[tk.u0];
  const int sx = u0.sx, sy = u0.sy;
  // Stage the tables.  Directions beyond the task's own are zero (they carry no flux); so is the whole table R, which
  // lanes outside the mesh read: their traces become zero, the vacuum inflow of the row they enter next.
  for (int e = threadIdx.x; e < (R + 1) * D * TW; e += blockDim.x) {
    const int k = e % TW, r = (e / TW) % (R + 1), d = e / (TW * (R + 1));
    tab[r * RS + 4 + ((d / VW) * TW + k) * VW + d % VW] =
        r < R && d < ndir ? reinterpret_cast<const T*>(a.linv)[(((size_t)tk.b * a.nu + tk.u0 + d) * R + r) * TW + k]
                          : (T)0;
  }
  for (int e = threadIdx.x; e < (R + 1) * 4; e += blockDim.x) {
    const int r = e >> 2;
    const T f = r < R ? ALG::factor(e & 3, (double)sx, (double)sy) : (T)0;
    tab[r * RS + (e & 3)] = a.sig_s && r < R ? f * reinterpret_cast<const T*>(a.sig_s)[(size_t)tk.b * R + r] : f;
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
  __syncthreads();
  if (warp >= W) return;
  const TI* src = reinterpret_cast<const TI*>(a.src) + in.off;
  T* part = reinterpret_cast<T*>(a.partial) + (size_t)a.tasks_per_inst * in.off + (size_t)tk.t * in.ndof;
  constexpr int YC = D * 2;   // elements per column of a trace buffer
  const T* yin = warp == 0 ? yfull : yring + (size_t)(warp - 1) * kRing * YC;
  T* yout = warp == W - 1 ? yfull : yring + (size_t)warp * kRing * YC;
  const unsigned yin_s = (unsigned)__cvta_generic_to_shared(yin);
  const int min_ = warp == 0 ? -1 : kRing - 1, mout = warp == W - 1 ? -1 : kRing - 1;
  const int cx = nx / a.rx, cy = ny / a.ry, dx = sx > 0 ? 1 : -1;
  const int P = wave_period(nx, W, SK);
  const int last = (nb - 1) / W;
  const int nsteps = last * P + (nb - 1 - last * W) * (32 + SK) + 31 + nx;
  const unsigned mx = 0xffffffffu / (unsigned)cx + 1u, my = 0xffffffffu / (unsigned)cy + 1u;   // i / c = mulhi(i, m); c = 1: see div
  auto div = [](int i, unsigned m) { return m ? (int)__umulhi((unsigned)i, m) : i; };
  const int rdx = sx > 0 ? RS : -RS, rowstep = 32 * RPL * W, dy = sy > 0 ? nx : -nx;
  auto cell0 = [&](int row) { return (sy > 0 ? row : ny - 1 - row) * nx + (sx > 0 ? 0 : nx - 1); };
  auto reg0 = [&](int row) {   // table of the row's first cell
    const int rr = div(row, my);
    return ((sy > 0 ? rr : a.ry - 1 - rr) * a.rx + (sx > 0 ? 0 : a.rx - 1)) * RS;
  };
  int row = 32 * RPL * warp + RPL * lane, col = -((32 + SK) * warp + lane);
  int cell = cell0(row), reg = reg0(row);
  int prow = row, pcol = col, pcell = cell;   // source prefetch, PF steps ahead
  auto fetch = [&](TI* dst) {
#pragma unroll
    for (int r = 0; r < RPL; ++r)
      if ((unsigned)pcol < (unsigned)nx && prow + r < ny)
        Vec4<TI>::load(src + 4 * (long long)(pcell + dx * pcol + r * dy), dst[4 * r], dst[4 * r + 1], dst[4 * r + 2],
                       dst[4 * r + 3]);
    ++pcol;
    const bool wrap = pcol == P;
    pcol = wrap ? 0 : pcol;
    prow = wrap ? prow + rowstep : prow;
    pcell = wrap ? pcell + (sy > 0 ? rowstep * nx : -rowstep * nx) : pcell;
  };
  TI q[PF][4 * RPL];
#pragma unroll
  for (int k = 0; k < PF; ++k) {
#pragma unroll
    for (int e = 0; e < 4 * RPL; ++e) q[k][e] = TI(0);
    fetch(q[k]);
  }
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
  // A double-float step is over a thousand instructions: unrolled, a group would not fit the instruction cache
  constexpr int UNR = std::is_same<T, dfloat>::value ? 1 : PF;
  for (int s0 = 0; s0 < nsteps; s0 += PF) {
#pragma unroll UNR
    for (int k0 = 0; k0 < PF; ++k0) {
      const int kk = UNR == 1 ? 0 : k0;
      const bool act = (unsigned)col < (unsigned)nx && row < ny;
      const int ro = act ? reg + rdx * div(col, mx) : R * RS;
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
      if constexpr (BC) {
#pragma unroll
        for (int v = 0; v < NV; ++v)
#pragma unroll
          for (int e = 0; e < 2; ++e)
#pragma unroll
            for (int r = 0; r < RPL; ++r)
              if (col == 0) X[r][v][e] = V::all(bx[e]);
      }
      const Blk<T, 4> sg = *reinterpret_cast<const Blk<T, 4>*>(tab + ro);
      V S[RPL][4], acc[RPL][4];
#pragma unroll
      for (int r = 0; r < RPL; ++r) {
        T t[4], Sr[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) t[e] = (T)q[kk][4 * r + e] * sg.v[e];
        ALG::to_basis(t, Sr);
#pragma unroll
        for (int e = 0; e < 4; ++e) S[r][e] = V::all(Sr[e]);
      }
      if constexpr (UNR == 1) {
#pragma unroll
        for (int k = 0; k + 1 < PF; ++k)
#pragma unroll
          for (int e = 0; e < 4 * RPL; ++e) q[k][e] = q[k + 1][e];
        fetch(q[PF - 1]);
      } else {
        fetch(q[kk]);
      }
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const Blk<V, TW> m = *reinterpret_cast<const Blk<V, TW>*>(tab + ro + 4 + v * TW * VW);
        if constexpr (kRegConst) {
#pragma unroll
          for (int r = 0; r < RPL; ++r) ALG::cell(S[r], X[r][v], Y[v], m.v, creg[v], acc[r], v == 0);
        } else {
          V c[NC];
#pragma unroll
          for (int e = 0; e < NC; ++e) c[e] = *reinterpret_cast<const V*>(cst + (v * NC + e) * VW);
#pragma unroll
          for (int r = 0; r < RPL; ++r) ALG::cell(S[r], X[r][v], Y[v], m.v, c, acc[r], v == 0);
        }
      }
#pragma unroll
      for (int r = 0; r < RPL; ++r) {
        T c4[4], o[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) c4[e] = acc[r][e].sum();
        ALG::from_basis(c4, o);
        o[1] = sx > 0 ? o[1] : -o[1];
        o[2] = sy > 0 ? o[2] : -o[2];
        o[3] = sx * sy > 0 ? o[3] : -o[3];
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
      ++col;
      const bool wrap = col == P;
      col = wrap ? 0 : col;
      row = wrap ? row + rowstep : row;
      cell = wrap ? cell + (sy > 0 ? rowstep * nx : -rowstep * nx) : cell;
      reg = wrap ? reg0(row) : reg;
    }
    group_sync(W);
  }
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

static size_t table_smem(const rte_problem* p, int prec, WaveShape s, int tw) {
  int nx, ny;
  mesh_max(p, &nx, &ny);
  const int nc = prec == PREC_F32 ? Rot<float>::NC : Modal<double>::NC;
  const int bytes = prec == PREC_F32 ? 4 : 8;
  const size_t elems = (size_t)(p->R + 1) * table_stride(4 + s.D * tw, bytes) + ((s.D * nc + 3) & ~3) +
                       ((size_t)nx + (s.W - 1) * kRing) * s.D * 2;
  return elems * bytes;
}

// FP64 tasks of one or two directions run in the Legendre basis while its tables (sixteen entries a direction and region)
// fit: up to about 1,300 regions with one direction, 750 with two.  The eigenbasis's four take twice as many and more.
static bool legendre(const rte_problem* p, int prec, WaveShape s) {
  return prec == PREC_F64 && s.D <= 2 && table_smem(p, prec, s, Legendre<double>::TW) <= kMaxSmem;
}

size_t wave_smem(const rte_problem* p, int prec, WaveShape s) {
  return table_smem(p, prec, s, prec == PREC_F32          ? Rot<float>::TW
                                : legendre(p, prec, s) ? Legendre<double>::TW
                                                       : Modal<double>::TW);
}

// Registers a thread of each built shape takes (0: not built): they set how many warps an SM holds.
static int shape_regs(int prec, int D, int rpl) {
  if (prec == PREC_F32) {
    if (rpl == 2) return D == 8 ? 208 : 0;
    switch (D) {
      case 1: return 96;
      case 2: return 112;
      case 4: case 8: return 128;
      case 12: return 200;
      case 16: return 224;
    }
    return 0;
  }
  if (rpl != 1) return 0;
  switch (D) {
    case 1: case 2: return 112;
    case 3: return prec == PREC_F64 ? 128 : 0;
    case 4: return 136;
    case 8: return prec == PREC_F64 ? 168 : 0;
  }
  return 0;
}

bool wave_shape_ok(const rte_problem* p, int prec, WaveShape s) {
  if (s.W < 1 || s.W > 8 || shape_regs(prec, s.D, s.rpl) == 0 || wave_smem(p, prec, s) > kMaxSmem) return false;
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
// two rows); FP64 19 cycles of the SM's FP64 unit for each of 24 D + 30 instructions (32 D + 4 in
// the Legendre basis; 5 % more a direction above 4), 70 alone; double-float 320 D + 264 instructions, 0.85 a cycle and SM quarter, 0.7 alone.  The partial fluxes, written and read once, are
// added at the copy bandwidth.
static double wave_cost(const rte_problem* p, int prec, WaveShape s, int sms, const std::vector<int>& order) {
  const int SK = 4, per_sm = 65536 / (shape_regs(prec, s.D, s.rpl) * 32);
  const size_t smem = wave_smem(p, prec, s) + 1024;
  const size_t slots = std::max(1, std::min(per_sm / s.W, (int)(kMaxSmem / smem)));
  int chunks = 0;
  for (int q = 0; q < 4; ++q) chunks += (p->quad_start[q + 1] - p->quad_start[q] + s.D - 1) / s.D;
  double pipe, alone;
  if (prec == PREC_F32) {
    pipe = (s.rpl == 2 ? 13.0 * s.D + 30.0 : 10.0 * s.D + 40.0) / (s.W == 1 ? 0.65 : 0.75);
    alone = s.rpl == 2 ? 1750.0 : 50.0 * s.D + 300.0;
  } else if (prec == PREC_F64) {
    const double instr = legendre(p, prec, s) ? 32.0 * s.D + 4.0 : 24.0 * s.D + 30.0;
    pipe = 19.0 * (1.0 + 0.05 * std::max(0, s.D - 4)) * instr;
    alone = 70.0 * instr;
  } else {
    pipe = (320.0 * s.D + 264.0) / 3.4;   // of warps in multiples of four
    alone = (320.0 * s.D + 264.0) / 0.7;
  }
  struct Run {
    double steps;
    int W;
  };
  std::vector<Run> queue, held;
  for (long long i = 0; i < (long long)p->B * chunks; i += sms) {
    const int b = order[i / chunks];
    const int nb = (p->ny[b] + 32 * s.rpl - 1) / (32 * s.rpl), W = std::min(s.W, nb), last = (nb - 1) / W;
    queue.push_back({(double)last * wave_period(p->nx[b], W, SK) + (nb - 1 - last * W) * (32 + SK) + 31 + p->nx[b], W});
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

template <typename T, typename TI, typename ALG, int VW, int NV, int RPL, int PF, bool BC, int MINB>
static int launch_one(const SweepArgs& a, int W, size_t smem, cudaStream_t st) {
  auto kern = k_wave<T, TI, ALG, VW, NV, RPL, PF, BC, MINB>;
  static std::atomic<size_t> granted[kMaxDevices];
  RTE_TRY(grant_smem(kern, smem, granted));
  kern<<<a.ntasks, W * 32, smem, st>>>(a);
  count_launch();
  RTE_CHECK_CUDA(cudaGetLastError());
  return RTE_OK;
}

// FP32 sweeps of FP64 vectors: the right-hand side, and the inner solves with FP64 Krylov vectors
template <typename TI>
static int launch_f32(const SweepArgs& a, WaveShape s, size_t smem, cudaStream_t st) {
  using A = Rot<float>;
  constexpr bool BC = std::is_same<TI, double>::value;
  switch (s.D * 10 + s.rpl) {
    case 11: return launch_one<float, TI, A, 1, 1, 1, 8, BC, 2>(a, s.W, smem, st);
    case 21: return launch_one<float, TI, A, 2, 1, 1, 8, BC, 2>(a, s.W, smem, st);
    case 41: return launch_one<float, TI, A, 2, 2, 1, 8, BC, 2>(a, s.W, smem, st);
    case 81: return launch_one<float, TI, A, 2, 4, 1, 4, BC, 2>(a, s.W, smem, st);
    case 121: return launch_one<float, TI, A, 2, 6, 1, 4, BC, 1>(a, s.W, smem, st);
    case 161: return launch_one<float, TI, A, 2, 8, 1, 4, BC, 1>(a, s.W, smem, st);
    case 82: return launch_one<float, TI, A, 2, 4, 2, 4, BC, 1>(a, s.W, smem, st);
  }
  set_error("sweep: unsupported directions per task");
  return RTE_ERR_UNSUPPORTED;
}

template <bool BC>
static int launch_f64(const SweepArgs& a, WaveShape s, bool leg, size_t smem, cudaStream_t st) {
  using A = Modal<double>;
  using Leg = Legendre<double>;
  switch (s.D) {
    case 1:
      return leg ? launch_one<double, double, Leg, 1, 1, 1, 4, BC, 2>(a, s.W, smem, st)
                 : launch_one<double, double, A, 1, 1, 1, 4, BC, 2>(a, s.W, smem, st);
    case 2:
      return leg ? launch_one<double, double, Leg, 1, 2, 1, 4, BC, 2>(a, s.W, smem, st)
                 : launch_one<double, double, A, 1, 2, 1, 4, BC, 2>(a, s.W, smem, st);
    case 3: return launch_one<double, double, A, 1, 3, 1, 4, BC, 2>(a, s.W, smem, st);
    case 4: return launch_one<double, double, A, 1, 4, 1, 4, BC, 1>(a, s.W, smem, st);
    case 8: return launch_one<double, double, A, 1, 8, 1, 4, BC, 1>(a, s.W, smem, st);
  }
  set_error("sweep: unsupported directions per task");
  return RTE_ERR_UNSUPPORTED;
}

static int launch_df(const SweepArgs& a, WaveShape s, size_t smem, cudaStream_t st) {
  using A = Modal<dfloat>;
  switch (s.D) {
    case 1: return launch_one<dfloat, dfloat, A, 1, 1, 1, 4, false, 2>(a, s.W, smem, st);
    case 2: return launch_one<dfloat, dfloat, A, 1, 2, 1, 4, false, 2>(a, s.W, smem, st);
    case 4: return launch_one<dfloat, dfloat, A, 1, 4, 1, 4, false, 1>(a, s.W, smem, st);
  }
  set_error("sweep: unsupported directions per task");
  return RTE_ERR_UNSUPPORTED;
}

int launch_wave(const rte_problem* p, int prec, WaveShape s, bool in64, const SweepArgs& args, cudaStream_t st) {
  SweepArgs a = args;
  if (prec == PREC_F32) a.linv = p->d_rot32.p;
  else if (prec == PREC_DF) a.linv = p->d_modal_df.p;
  const bool leg = legendre(p, prec, s);
  if (prec == PREC_F64) a.linv = leg ? p->d_linv64.p : p->d_modal64.p;
  if (!wave_shape_ok(p, prec, s)) {
    set_error("sweep: shared-memory table too large for this mesh/region count");
    return RTE_ERR_UNSUPPORTED;
  }
  const size_t smem = wave_smem(p, prec, s);
  if (prec == PREC_F64)
    return a.with_bc ? launch_f64<true>(a, s, leg, smem, st) : launch_f64<false>(a, s, leg, smem, st);
  if (prec == PREC_DF) return launch_df(a, s, smem, st);
  return in64 ? launch_f32<double>(a, s, smem, st) : launch_f32<float>(a, s, smem, st);
}

}  // namespace rte
